"""What the FP64 hop computes outside its fixed-point format does not depend on how many sites of a warp need that: up to
four are taken one after another by four pairs of lanes, more by a lane each."""
import numpy as np
import pytest

from gpu_util import gpu_dslash, make_context, seeded_gauge
from oracle import lattice
from paper_1710_09178_gb300 import inputs

pytestmark = pytest.mark.gpu

FP64 = 0


@pytest.mark.parametrize("dims", [(16, 4, 4, 4), (6, 6, 2, 2)])  # V/2 = 512; 72: the last group has 8 sites
@pytest.mark.parametrize("first", [0, 32, 64])
def test_one_site_among_many(dims, first):
    U, psi = seeded_gauge(dims, 3), inputs.gaussian_vector(dims, 21)
    even = np.flatnonzero(lattice.parity(dims) == 0)
    size = min(32, len(even) - first)
    base = gpu_dslash(make_context(dims, 0.1, U=U)[0], psi, 0, FP64)
    one = None
    for n in (1, 2, 4, 5, 31, 32):
        if n > size:
            continue
        W = U.copy()
        W[even[first:first + n], 1] *= 7  # forward links: each in the sum of its own site only, and outside the format
        got = gpu_dslash(make_context(dims, 0.1, U=W)[0], psi, 0, FP64)
        one = got[first] if one is None else one
        assert np.array_equal(got[first], one)
        rest = np.r_[0:first, first + n:len(even)]
        assert np.array_equal(got[rest], base[rest])
        assert np.all(np.abs(got[first:first + n] - base[first:first + n]).max(1) > 0)
