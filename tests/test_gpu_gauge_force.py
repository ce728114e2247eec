"""The gauge force holds every component to FP64 accuracy, however small it is beside the links' other entries.

One Omelyan step of length h = 2^-40 with lambda = 1/2 and an action without pseudofermion leaves the momenta
-h (F(U0) + F(U1)) / 2, U1 the links it returns (the links move by rounding only).

Bar, per component: 36 x 2^-53 of the sum of the magnitudes of the products of links that make it up: 24 for U A (three
products of up to 6 roundings, six staples added), the rest for the traceless part, the factors and the kicks.  The reference is
long double."""
import numpy as np
import pytest

from gpu_util import make_context, to_dev
from oracle import force, lattice
from paper_1710_09178_gb300 import inputs

pytestmark = pytest.mark.gpu

DIMS, BETA, H = (4, 4, 2, 6), 5.4, 2.0 ** -40
BAR = 36 * 2.0 ** -53


def exact_force(U):
    """Components of the gauge force and their magnitudes, (V, 4, 8) long double."""
    W, S = [], []
    dag = lambda M: M.conj().swapaxes(-1, -2)
    absr = lambda M: np.block([[abs(M.real), abs(M.imag)], [abs(M.imag), abs(M.real)]]).astype(np.float64)
    U = U.astype(np.clongdouble)
    for mu in range(4):
        up = lattice.neighbour(DIMS, mu, +1)
        w = s = 0
        for nu in set(range(4)) - {mu}:
            vp, vm = lattice.neighbour(DIMS, nu, +1), lattice.neighbour(DIMS, nu, -1)
            for a, b, c in ((U[up, nu], dag(U[vp, mu]), dag(U[:, nu])), (dag(U[vm[up], nu]), dag(U[vm, mu]), U[vm, nu])):
                w = w + a @ b @ c
                s = s + absr(a) @ absr(b) @ absr(c)
        W.append(U[:, mu] @ w)
        S.append(absr(U[:, mu]) @ s)
    W, S = np.stack(W, 1), np.stack(S, 1)
    re, im, sre, sim = W.real, W.imag, S[..., :3, :3], S[..., :3, 3:]
    F, M = np.zeros(W.shape[:2] + (8,), np.longdouble), np.zeros(W.shape[:2] + (8,))
    for a, r, c in ((0, 0, 1), (3, 0, 2), (5, 1, 2)):
        F[..., a], M[..., a] = im[..., r, c] + im[..., c, r], sim[..., r, c] + sim[..., c, r]
        F[..., a + 1], M[..., a + 1] = re[..., r, c] - re[..., c, r], sre[..., r, c] + sre[..., c, r]
    F[..., 2] = im[..., 0, 0] - im[..., 1, 1]
    F[..., 7] = (im[..., 0, 0] + im[..., 1, 1] - 2 * im[..., 2, 2]) / np.sqrt(np.longdouble(3))
    M[..., 2] = M[..., 7] = sim[..., 0, 0] + sim[..., 1, 1] + 2 * sim[..., 2, 2]
    return BETA / 6 * F, BETA / 6 * M


def near_one(eps, seed=9):
    """exp(i eps H), each entry to FP64 accuracy."""
    h = np.random.default_rng(seed).standard_normal((int(np.prod(DIMS)), 4, 8))
    X = 0.5j * eps * np.einsum("lma,aij->lmij", h, force.gell_mann())
    U = term = np.broadcast_to(np.eye(3, dtype=np.complex128), X.shape)
    for k in range(1, 20):
        term = term @ X / k
        U = U + term
    return U


def links(kind):
    U = inputs.gauge_field(DIMS, seed=3)
    if kind == "unit":
        U = np.broadcast_to(np.eye(3, dtype=np.complex128), U.shape).copy()
    elif kind == "blocks":  # SU(2) in colours 0 and 1
        n = np.random.default_rng(5).standard_normal(U.shape[:2] + (4,))
        n /= np.linalg.norm(n, axis=-1, keepdims=True)
        U = np.zeros_like(U)
        U[..., 0, 0], U[..., 0, 1] = n[..., 0] + 1j * n[..., 1], n[..., 2] + 1j * n[..., 3]
        U[..., 1, 0], U[..., 1, 1] = -U[..., 0, 1].conj(), U[..., 0, 0].conj()
        U[..., 2, 2] = 1
    elif kind == "mixed":  # rough beside smooth
        U[::3] = near_one(1e-6)[::3]
    elif kind != "rough":
        U = near_one(float(kind))
    return U


@pytest.mark.parametrize("kind", ["rough", "0.3", "0.1", "1e-3", "1e-9", "unit", "blocks", "mixed"])
def test_every_component_is_accurate(kind):
    import torch

    import paper_1710_09178_gb300 as lq

    U0 = links(kind)
    V = len(U0)
    ctx, _ = make_context(DIMS, 0.1, U=U0)
    Ud, P0 = to_dev(U0), torch.zeros((V, 4, 8), dtype=torch.float64, device="cuda")
    mom, U1 = torch.empty_like(P0), torch.empty_like(Ud)
    rc, _ = lq.rhmc_trajectory(ctx, Ud, P0, to_dev(inputs.gaussian_vector(DIMS, 4)), 0.0, BETA, H, 1,
                               (0.0, [0.0], [1.0]), tol=1e-8, prec=lq.FP64, phi_given=True, mom_out=mom, links_out=U1,
                               lam=0.5)
    assert rc == 0
    U1 = U1.cpu().numpy()
    assert np.max(np.abs(U1 - U0)) <= 1e-14
    (F0, S0), (F1, S1) = exact_force(U0), exact_force(U1)
    err = np.abs(mom.cpu().numpy() / -H - (F0 + F1) / 2)
    assert np.all(err <= BAR * (S0 + S1) / 2), float(np.max(err / np.maximum((S0 + S1) / 2, 1e-300)) * 2 ** 53)
