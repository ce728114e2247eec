"""The sizes where the Dslash and the solver change kernels: lattices of exactly 152 blocks of 128 sites (all loads
at once and the folded p update up to there), 304 blocks of 32 or 64 double-FP32 sites, one block with a tail, and one
step beyond.

Bars: hops against the oracle as in the Dslash parity tests (FP32 2e-6, double-FP32 1e-13 relative); a solve of one source,
whose p update is folded on the small lattices, equals the same source of a multi-RHS solve, whose p update never is, bit
for bit."""
import numpy as np
import pytest

from gpu_util import gpu_dslash, make_context, rel_max, seeded_gauge, to_dev
from oracle import staggered
from paper_1710_09178_gb300 import inputs

pytestmark = pytest.mark.gpu

FP32, FP32_R12, FP16FIX, FP32_L16, DF64 = 1, 2, 3, 5, 6
# V/2 = 8, 240, 9728 = 304 x 32, 9760, 19456 = 152 x 128 = 304 x 64, 19520
DIMS = [(2, 2, 2, 2), (6, 4, 2, 10), (38, 16, 8, 4), (2, 10, 122, 8), (38, 16, 8, 8), (2, 16, 122, 10)]


@pytest.mark.parametrize("dims", DIMS)
def test_hops_match_oracle(dims):
    ctx, U = make_context(dims, 0.1, gauge_seed=3)
    psi = inputs.gaussian_vector(dims, 21)
    for p in (0, 1):
        ref = staggered.dslash_eo(U, psi, dims, p)
        for prec, bar in ((FP32, 2e-6), (FP32_R12, 2e-6), (DF64, 1e-13)):
            assert rel_max(gpu_dslash(ctx, psi, p, prec), ref) < bar


@pytest.mark.parametrize("dims,prec", [(d, FP32) for d in DIMS] + [((6, 4, 2, 10), q) for q in (FP32_R12, FP16FIX, FP32_L16)]
                         + [((38, 16, 8, 8), FP32_R12)])
@pytest.mark.parametrize("graph", [0, 1])
def test_folded_p_update_gives_the_same_bits(dims, prec, graph):
    import torch

    import paper_1710_09178_gb300 as lq

    mass = 0.1
    c0, res, poles, _ = lq.rational_coeffs(-0.5, 4 * mass ** 2, 16 + 4 * mass ** 2, 6)
    b = [to_dev(inputs.gaussian_vector(dims, 30 + s)) for s in range(2)]
    out = []
    for multi in (False, True):
        ctx = lq.Context(dims, mass)
        ctx.set_gauge(to_dev(seeded_gauge(dims, 3)))
        ctx.set_option(lq.OPT_USE_GRAPH, graph)
        xs = [[torch.empty_like(v) for _ in poles] for v in b]
        if multi:
            rc, st = lq.mshift_cg_multi(ctx, poles, res, c0, b, xs, None, tol=1e-9, prec=prec)
            st = st[0]
        else:
            rc, st = lq.mshift_cg(ctx, poles, res, c0, b[0], xs[0], None, tol=1e-9, prec=prec)
        torch.cuda.synchronize()
        assert rc == 0
        out.append((st["iterations"], st["shift_iterations"], [x.cpu().numpy() for x in xs[0]]))
    assert out[0][:2] == out[1][:2]
    assert all(np.array_equal(x, y) for x, y in zip(out[0][2], out[1][2]))
