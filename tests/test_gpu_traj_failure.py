"""A trajectory that fails after its links have moved leaves every link copy of the context on the moved links.

The start is the unit field, on which the shifted CG ends after about ten iterations (few distinct eigenvalues); half a
step of unit momenta makes the links rough, and the next force's solve runs into maxiter."""
import numpy as np
import pytest

from gpu_util import make_context, to_dev
from oracle import rational
from paper_1710_09178_gb300 import inputs

pytestmark = pytest.mark.gpu


def test_copies_are_current_after_a_failure_between_the_steps():
    import torch

    import paper_1710_09178_gb300 as lq

    dims, mass = (4, 4, 4, 6), 0.1
    act = rational.zolotarev_inv_sqrt(8, 4 * mass ** 2, 16 + 4 * mass ** 2)[:3]
    V = int(np.prod(dims))
    U0 = np.broadcast_to(np.eye(3, dtype=np.complex128), (V, 4, 3, 3)).copy()
    ctx, _ = make_context(dims, mass, U=U0)
    Ud = to_dev(U0)
    p0 = to_dev(inputs.counter_normal_pairs(32, np.arange(4 * V, dtype=np.uint64), 4).reshape(V, 4, 8))
    xi = to_dev(inputs.gaussian_vector(dims, 33))
    formats = (lq.FP64, lq.FP32, lq.FP32_R12, lq.FP32_R8, lq.FP32_L16, lq.DF64)

    def hops():
        out = []
        for prec in formats:
            vin, vout = ctx.new_vector(prec), ctx.new_vector(prec)
            ctx.pack(vin, prec, xi)
            lq.dslash_eo(ctx, vout, vin, 1, prec)
            r = torch.empty_like(xi)
            ctx.unpack(r, vout, prec)
            out.append(r.cpu().numpy())
        return out

    before = hops()
    rc, _ = lq.rhmc_trajectory(ctx, Ud, p0, xi, 0.0, 5.4, 1.0, 1, act, tol=1e-8, maxiter=40, prec=lq.FP32,
                               prec_action=lq.FP32, phi_given=True, raise_on_error=False)
    assert rc == lq.LQCD_ERR_NOT_CONVERGED
    assert np.array_equal(Ud.cpu().numpy(), U0)
    after = hops()
    size = np.max(np.abs(after[0]))
    assert np.max(np.abs(after[0] - before[0])) > 0.1 * size  # the links have moved
    for prec, a in zip(formats, after):
        # each format's hop within its own link precision of the FP64 one
        tol = {lq.FP32_R8: 1e-4, lq.FP32_L16: 2e-4}.get(prec, 2e-6)
        assert np.max(np.abs(a - after[0])) <= tol * size, prec
