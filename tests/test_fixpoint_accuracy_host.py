"""What the block fixed point of the FP64 half Dslash (csrc/fixpoint.h) accepts is as accurate as FP64 multiply-adds
(tests/native/fixpoint_accuracy_main.cpp)."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_accepted_sums_are_accurate(tmp_path):
    exe = tmp_path / "accuracy"
    r = subprocess.run(["g++", "-std=c++17", "-O1", "-Wall", "-Wextra", "-Werror", "-fsanitize=undefined",
                        "-fno-sanitize-recover", "-I" + os.path.join(ROOT, "paper_1710_09178_gb300", "csrc"),
                        os.path.join(ROOT, "tests", "native", "fixpoint_accuracy_main.cpp"), "-o", str(exe)],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0 and r.stdout.strip() == "ok", r.stdout + r.stderr
