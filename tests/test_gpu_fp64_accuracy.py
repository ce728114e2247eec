"""The FP64 hop holds every component to FP64 accuracy, however small it is beside the others.

Bar, per real component: 22 x 2^-53 of S, the sum of the magnitudes of its 48 products.  An FP64 sum in the order of
the kernel's fallback takes at most 11 roundings.  The block fixed point is used where its error is below 21 x 2^-53 S
(csrc/fixpoint.h), and is rounded to FP64 once.  The reference sums are long double (error below 2^-58 S)."""
import numpy as np
import pytest

from gpu_util import gpu_apply_A, gpu_dslash, make_context, seeded_gauge
from oracle import lattice
from paper_1710_09178_gb300 import inputs

pytestmark = pytest.mark.gpu

FP64 = 0
BAR = 22 * 2.0 ** -53


def exact_hop(U, psi, dims, p):
    """(D psi) on parity p and S, both as (Vh, 3, 2) long double (last axis: real, imaginary)."""
    fwd, bwd, sf, sb = lattice.neighbour_tables(dims)
    sites = [np.flatnonzero(lattice.parity(dims) == q) for q in (0, 1)]
    W = U.view(np.float64).reshape(-1, 4, 3, 3, 2).astype(np.longdouble)
    v = psi.view(np.float64).reshape(-1, 3, 2).astype(np.longdouble)
    out = np.zeros((len(psi), 3, 2), np.longdouble)
    mag = np.zeros_like(out)
    for mu in range(4):
        for j, M, sign in ((fwd[p][mu], W[sites[p], mu], sf[p][mu]),
                           (bwd[p][mu], W[sites[1 - p][bwd[p][mu]], mu].swapaxes(1, 2) * np.array([1, -1]), -sb[p][mu])):
            x = v[j][:, None]
            terms = np.stack([M[..., 0] * x[..., 0], -M[..., 1] * x[..., 1], M[..., 0] * x[..., 1], M[..., 1] * x[..., 0]], -1)
            h = 0.5 * np.asarray(sign)[:, None, None]
            out += h * np.stack([terms[..., :2].sum((-1, -2)), terms[..., 2:].sum((-1, -2))], -1)
            mag += 0.5 * np.abs(np.stack([np.abs(terms[..., :2]).sum((-1, -2)), np.abs(terms[..., 2:]).sum((-1, -2))], -1))
    return out, mag


def gauge(kind, dims):
    U = seeded_gauge(dims, 3).copy()
    if kind == "unit":
        U[:] = np.eye(3)
    elif kind == "blocks":  # SU(2) in colours 0 and 1
        n = np.random.default_rng(5).standard_normal(U.shape[:2] + (4,))
        n /= np.linalg.norm(n, axis=-1, keepdims=True)
        U[:] = 0
        U[..., 0, 0], U[..., 0, 1] = n[..., 0] + 1j * n[..., 1], n[..., 2] + 1j * n[..., 3]
        U[..., 1, 0], U[..., 1, 1] = -U[..., 0, 1].conj(), U[..., 0, 0].conj()
        U[..., 2, 2] = 1
    elif kind == "smooth":  # rotations by 1e-9: tiny off-diagonal entries
        U[:] = np.eye(3) + 1e-9 * (U - U.swapaxes(-1, -2).conj())
    elif kind == "small":
        U *= 1e-6
    return U


@pytest.mark.parametrize("kind", ["rough", "unit", "blocks", "smooth", "small"])
@pytest.mark.parametrize("colours", [(1, 1, 1), (1, 1e-12, 1e-20), (1e-9, 1, 0), (0, 0, 1)])
def test_every_component_is_accurate(kind, colours):
    dims = (10, 6, 4, 6)
    U, psi = gauge(kind, dims), inputs.gaussian_vector(dims, 21) * np.array(colours)
    if colours[2] == 0:  # real and imaginary parts of different size too
        psi = psi.real + 1e-15j * psi.imag
    ctx, _ = make_context(dims, 0.1, U=U)
    for p in (0, 1):
        want, mag = exact_hop(U, psi, dims, p)
        got = gpu_dslash(ctx, psi, p, FP64).view(np.float64).reshape(-1, 3, 2)
        assert np.all(np.abs(got - want) <= BAR * mag)


def test_operator_and_spread_vectors():
    # components over 24 orders of magnitude; A = 4 m^2 - D_eo D_oe with both hops of it
    dims, mass = (10, 6, 4, 6), 0.1
    U, psi = gauge("rough", dims), inputs.gaussian_vector(dims, 22)
    psi = psi * 10.0 ** np.random.default_rng(4).uniform(-12, 12, psi.shape)
    ctx, _ = make_context(dims, mass, U=U)
    for p in (0, 1):
        want, mag = exact_hop(U, psi, dims, p)
        got = gpu_dslash(ctx, psi, p, FP64).view(np.float64).reshape(-1, 3, 2)
        assert np.all(np.abs(got - want) <= BAR * mag)
    unit = gauge("unit", dims)
    psi = inputs.gaussian_vector(dims, 23) * np.array([1, 1e-12, 1e-20])
    ctx, _ = make_context(dims, mass, U=unit)
    odd, modd = exact_hop(unit, psi, dims, 1)
    rounded = (odd[..., 0] + 1j * odd[..., 1]).astype(np.complex128)
    even, meven = exact_hop(unit, rounded, dims, 0)
    _, spread = exact_hop(unit, (modd[..., 0] + 1j * modd[..., 1]).astype(np.complex128), dims, 0)
    v = psi.view(np.float64).reshape(-1, 3, 2)
    got = gpu_apply_A(ctx, psi, 0.0, FP64)[0].view(np.float64).reshape(-1, 3, 2)
    # the inner hop's errors spread by the outer one; two roundings for 4 m^2 psi and the difference
    bar = BAR * (meven + 2 * spread) + 2.0 ** -52 * (np.abs(4 * mass ** 2 * v) + np.abs(even))
    assert np.all(np.abs(got - (4 * mass ** 2 * v - even)) <= bar)
