"""rhmc_trajectory against the oracle trajectory where its gauge force and link update can go wrong: extents of 2
(a site is its own neighbour's neighbour), a ragged lattice, links outside the fixed-point format (computed in
FP64), and steps long enough for the exponential's squaring (|h P| > 1/4, several times).

Bars: those of the trajectory parity tests (FP64 solves to 1e-12): Hamiltonian pieces 1e-9 relative, links and
momenta 1e-8; momenta scaled by their size (they grow with the force of the longer steps)."""
import numpy as np
import pytest

from gpu_util import make_context, to_dev
from oracle import rational, rhmc
from paper_1710_09178_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims,tau,nsteps,factor", [
    ((2, 2, 2, 2), 0.3, 3, 1.0),
    ((6, 4, 2, 10), 0.2, 2, 1.0),
    ((4, 4, 4, 4), 0.3, 3, 1.2),
    ((4, 4, 4, 4), 0.6, 1, 1.0),
])
def test_trajectory_matches_oracle(dims, tau, nsteps, factor):
    import torch

    import paper_1710_09178_gb300 as lq

    mass, beta = 0.1, 5.4
    lo, hi = 4 * mass ** 2, 16 + 4 * mass ** 2
    act, heat = rational.zolotarev_inv_sqrt(8, lo, hi)[:3], rational.remez_power(0.25, lo, hi, 8)[:3]
    V = int(np.prod(dims))
    U0 = inputs.gauge_field(dims, seed=31)
    U0[V // 3, 2] *= factor  # one link off SU(3)
    p0 = inputs.counter_normal_pairs(32, np.arange(4 * V, dtype=np.uint64), 4).reshape(V, 4, 8)
    xi = inputs.gaussian_vector(dims, 33)
    ctx, _ = make_context(dims, mass, U=U0)
    Ud = to_dev(U0)
    links, mom = torch.empty_like(Ud), torch.empty((V, 4, 8), dtype=torch.float64, device="cuda")
    rc, res = lq.rhmc_trajectory(ctx, Ud, to_dev(p0), to_dev(xi), 0.5, beta, tau, nsteps, act, heat, tol=1e-12,
                                 prec=lq.FP64, mom_out=mom, links_out=links)
    assert rc == 0
    Uo, acc, info = rhmc.trajectory(U0, p0, xi, 0.5, dims, mass, beta, tau, nsteps, act, heat, tol=1e-12)
    for k in ("kinetic", "gauge", "fermion"):
        for end, parts in (("0", info["parts0"]), ("1", info["parts1"])):
            assert abs(res[k + end] - parts[k]) <= 1e-9 * max(abs(parts[k]), 1.0)
    assert np.max(np.abs(links.cpu().numpy() - info["U1"])) <= 1e-8
    assert np.max(np.abs(mom.cpu().numpy() - info["p1"])) <= 1e-8 * max(1.0, np.max(np.abs(info["p1"])))


@pytest.mark.parametrize("uniform,maxiter", [(0.0, 20000), (1e9, 20000), (0.0, 40)])  # accepted, rejected, failed inside
def test_every_link_copy_is_current_after_a_trajectory(uniform, maxiter):
    # the compact copies are left out while the links move: afterwards each format's hop equals that of a fresh
    # context holding the same links, bit for bit (a failed trajectory leaves links of its own, in every copy)
    import torch

    import paper_1710_09178_gb300 as lq

    dims, mass = (4, 4, 4, 6), 0.1
    lo, hi = 4 * mass ** 2, 16 + 4 * mass ** 2
    act, heat = rational.zolotarev_inv_sqrt(8, lo, hi)[:3], rational.remez_power(0.25, lo, hi, 8)[:3]
    V = int(np.prod(dims))
    ctx, U0 = make_context(dims, mass, gauge_seed=31)
    Ud = to_dev(U0)
    p0 = to_dev(inputs.counter_normal_pairs(32, np.arange(4 * V, dtype=np.uint64), 4).reshape(V, 4, 8))
    xi = to_dev(inputs.gaussian_vector(dims, 33))
    rc, res = lq.rhmc_trajectory(ctx, Ud, p0, xi, uniform, 5.4, 0.3, 3, act, heat, tol=1e-8, maxiter=maxiter,
                                 prec=lq.FP32, raise_on_error=False)
    formats = (lq.FP64, lq.FP32, lq.FP32_R12, lq.FP32_R8, lq.FP32_L16, lq.DF64)

    def hops(c):
        out = []
        for prec in formats:
            vin, vout = c.new_vector(prec), c.new_vector(prec)
            c.pack(vin, prec, xi)
            lq.dslash_eo(c, vout, vin, 1, prec)
            r = torch.empty_like(xi)
            c.unpack(r, vout, prec)
            out.append(r.cpu().numpy())
        return out

    got = hops(ctx)
    if rc == 0:
        assert res["accepted"] == (uniform == 0.0)
        fresh = lq.Context(dims, mass)
        fresh.set_gauge(Ud)
        for prec, a, b in zip(formats, got, hops(fresh)):
            assert np.array_equal(a, b), prec
    else:
        # all copies hold one field: every format's hop is within its own link precision of the FP64 one
        for prec, a in zip(formats, got):
            tol = {lq.FP32_R8: 1e-4, lq.FP32_L16: 2e-4}.get(prec, 2e-6)
            assert np.max(np.abs(a - got[0])) <= tol * np.max(np.abs(got[0])), prec
