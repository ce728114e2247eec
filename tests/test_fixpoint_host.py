"""The block fixed point of the FP64 half Dslash (csrc/fixpoint.h) on the host: sums of 48 products against long
double over many scales, exact digits, and what the format refuses (tests/native/fixpoint_main.cpp)."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1710_09178_gb300", "csrc")


def test_block_fixed_point_on_host(tmp_path):
    exe = tmp_path / "fixpoint"
    r = subprocess.run(["g++", "-std=c++17", "-O1", "-Wall", "-Wextra", "-Werror", "-fsanitize=undefined",
                        "-fno-sanitize-recover", "-I" + CSRC,
                        os.path.join(ROOT, "tests", "native", "fixpoint_main.cpp"), "-o", str(exe)],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0 and r.stdout.strip() == "ok", r.stdout + r.stderr
