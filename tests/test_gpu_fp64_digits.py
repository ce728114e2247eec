"""No result depends on whether a context keeps the digits of its FP64 links (LQCD_OPT_FP64_DIGITS, and by itself where
memory is short): the same bits with and without, for every entry point that reads them."""
import numpy as np
import pytest

from gpu_util import seeded_gauge, to_dev
from oracle import rational
from paper_1710_09178_gb300 import inputs

pytestmark = pytest.mark.gpu


def links(kind, dims):
    U = seeded_gauge(dims, 3).copy()
    if kind == "off":  # some links outside the format, one of them not finite
        U[5, 2] *= 7
        U[11, 0] *= 1e3
        U[12, 1, 2, 2] = np.inf
    elif kind == "sizes":  # entries of all sizes
        U *= 10.0 ** np.random.default_rng(2).uniform(-30, 0, U.shape)
    elif kind == "scaled":
        U *= 1.2
    return U


def contexts(U, dims, mass=0.1):
    import paper_1710_09178_gb300 as lq

    out = []
    for digits in (1, 0):
        ctx = lq.Context(dims, mass)
        ctx.set_option(lq.OPT_FP64_DIGITS, digits)
        ctx.set_gauge(to_dev(U))
        with pytest.raises(lq.LqcdError):  # chosen before the first field
            ctx.set_option(lq.OPT_FP64_DIGITS, digits)
        out.append(ctx)
    return out


def same(a, b):
    return np.array_equal(a.cpu().numpy(), b.cpu().numpy(), equal_nan=True)


@pytest.mark.parametrize("kind", ["rough", "off", "sizes", "scaled"])
@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (10, 6, 4, 6), (16, 16, 16, 12)])
def test_hop_operator_and_batch(dims, kind):
    import torch

    import paper_1710_09178_gb300 as lq

    if kind == "off" and dims == (2, 2, 2, 2):
        pytest.skip("16 sites: too few links")
    psi = to_dev(inputs.gaussian_vector(dims, 21))
    got = []
    ctxs = contexts(links(kind, dims), dims)
    vecs = []
    for ctx in ctxs:
        vin, vout, vq = (ctx.new_vector(lq.FP64) for _ in range(3))
        ctx.pack(vin, lq.FP64, psi)
        r = []
        for p in (0, 1):
            lq.dslash_eo(ctx, vout, vin, p, lq.FP64)
            r.append(vout.view(torch.float64).clone())
        dot = ctx.apply_A(vq, vin, 0.3, lq.FP64, want_dot=True)
        r.append(vq.view(torch.float64).clone())
        r.append(torch.tensor([dot]))
        got.append(r)
        vecs.append((vin, vout))
    assert all(same(a, b) for a, b in zip(*got))
    # a batch of both kinds of contexts, then of one kind
    for pick in ((0, 1), (1, 0), (0,), (1,)):
        outs = [ctxs[k].new_vector(lq.FP64) for k in pick]
        lq.dslash_eo_batch([ctxs[k] for k in pick], outs, [vecs[k][0] for k in pick], [1] * len(pick), lq.FP64)
        assert all(same(o.view(torch.float64), got[0][1]) for o in outs)


def test_solve_force_and_trajectory():
    import torch

    import paper_1710_09178_gb300 as lq

    dims, mass = (4, 4, 4, 6), 0.1
    lo, hi = 4 * mass ** 2, 16 + 4 * mass ** 2
    act, heat = rational.zolotarev_inv_sqrt(8, lo, hi)[:3], rational.remez_power(0.25, lo, hi, 8)[:3]
    V = int(np.prod(dims))
    U = links("rough", dims)
    U[V // 3, 2] *= 1.2  # one link off SU(3)
    U[V // 2] = np.eye(3)  # smooth ones beside rough ones
    p0 = to_dev(inputs.counter_normal_pairs(32, np.arange(4 * V, dtype=np.uint64), 4).reshape(V, 4, 8))
    xi = to_dev(inputs.gaussian_vector(dims, 33))
    got = []
    for ctx in contexts(U, dims, mass):
        xs, y = [torch.empty_like(xi) for _ in act[2]], torch.empty_like(xi)
        F = torch.empty((V, 4, 8), dtype=torch.float64, device="cuda")
        assert lq.mshift_cg(ctx, act[2], act[1], act[0], xi, xs, y, tol=1e-10, prec=lq.FP64)[0] == 0
        assert lq.fermion_force(ctx, act[2], act[1], act[0], xi, Falg=F, tol=1e-10, prec=lq.FP64)[0] == 0
        Ud = to_dev(U)
        links_out, mom = torch.empty_like(Ud), torch.empty_like(p0)
        rc, res = lq.rhmc_trajectory(ctx, Ud, p0, xi, 0.5, 5.4, 0.2, 2, act, heat, tol=1e-10, prec=lq.FP64,
                                     mom_out=mom, links_out=links_out)
        assert rc == 0
        got.append(xs + [y, F, links_out, mom, torch.tensor([res["H0"], res["H1"]])])
    assert all(same(a, b) for a, b in zip(*got))
