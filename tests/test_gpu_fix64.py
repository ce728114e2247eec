"""The FP64 half Dslash in block fixed point against the FP64 oracle where the format can go wrong: group
tails, lattices of several groups per block, zeros, wide scales, and what has to be computed in FP64 instead.

Bar: an FP64 sum of 48 products rounds by at most 48 x 2^-53 x 9.82 = 5.3e-14 of the largest neighbouring component
(8 row norms of 1/2 times sqrt(6)); the oracle is such a sum, the fixed-point sum errs by less."""
import numpy as np
import pytest

from gpu_util import gpu_dslash, make_context, seeded_gauge
from oracle import lattice, staggered
from paper_1710_09178_gb300 import inputs

pytestmark = pytest.mark.gpu

FP64 = 0
BAR = 5.3e-14


def check(dims, U, psi, scale=1.0):
    ctx, _ = make_context(dims, 0.1, U=U)
    fwd, bwd, _, _ = lattice.neighbour_tables(dims)
    for p in (0, 1):
        ref = staggered.dslash_eo(U, psi, dims, p)
        got = gpu_dslash(ctx, psi, p, FP64)
        # what is infinite or NaN follows from the products' order, that it is not finite does not
        assert np.array_equal(np.isfinite(got), np.isfinite(ref))
        big = np.abs(psi.view(np.float64).reshape(len(psi), 6)).max(1)
        near = np.maximum(big[fwd[p]].max(0), big[bwd[p]].max(0))  # largest neighbouring component per site
        fine = np.isfinite(near) & np.isfinite(ref).all(1)
        err = np.abs(got - ref).view(np.float64).reshape(len(psi), -1).max(1)
        assert np.all(err[fine] <= BAR * scale * near[fine])


# V/2 = 8: less than a group; 48 and 720: ragged tails; 15360: two groups in some blocks; 16^3x12: several in all
@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (6, 4, 2, 2), (10, 6, 4, 6), (16, 16, 12, 10), (16, 16, 16, 12)])
def test_sizes(dims):
    check(dims, seeded_gauge(dims, 3), inputs.gaussian_vector(dims, 21))


@pytest.mark.parametrize("case", ["sites", "components", "point", "tiny", "huge", "denormal", "nan", "inf", "beyond"])
def test_vector_scales(case):
    dims = (10, 6, 4, 6)
    psi = inputs.gaussian_vector(dims, 22)
    rng = np.random.default_rng(4)
    if case == "sites":
        psi = psi * 10.0 ** rng.uniform(-15, 15, (len(psi), 1))
    elif case == "components":
        psi = psi * 10.0 ** rng.uniform(-12, 12, psi.shape)
    elif case == "point":
        psi = np.zeros_like(psi)
        psi[100, 2] = 1 - 2j
    elif case == "beyond":  # neighbours on both sides of the format's limits
        psi = psi * 10.0 ** rng.uniform(-260, 260, (len(psi), 1))
    elif case in ("tiny", "huge", "denormal"):
        psi = psi * {"tiny": 1e-280, "huge": 1e280, "denormal": 1e-310}[case]
    else:
        psi[77, 1] = np.nan if case == "nan" else np.inf
    if case == "denormal":  # the oracle's products round to multiples of 2^-1074
        ctx, U = make_context(dims, 0.1, gauge_seed=3)
        for p in (0, 1):
            ref = staggered.dslash_eo(U, psi, dims, p)
            assert np.abs(gpu_dslash(ctx, psi, p, FP64) - ref).max() <= 96 * 2.0 ** -1074
        return
    with np.errstate(all="ignore"):
        check(dims, seeded_gauge(dims, 3), psi)


@pytest.mark.parametrize("factor", [7.0, 1e3, 1e-3, 0.0, np.nan])
def test_links_outside_the_format(factor):
    # one link, then all of them, scaled: rows of norm above 1/2 are computed in FP64, smaller ones are not
    dims = (10, 6, 4, 6)
    U = seeded_gauge(dims, 3).copy()
    U[5, 2] = U[5, 2] * factor
    with np.errstate(all="ignore"):
        check(dims, U, inputs.gaussian_vector(dims, 23), scale=max(1.0, abs(factor)) if factor == factor else 1.0)
        if factor == factor:
            check(dims, seeded_gauge(dims, 3) * factor, inputs.gaussian_vector(dims, 24), scale=max(1.0, abs(factor)))
