"""Moments at the edges of the reduction: parts of a warp, whole warps, a whole block and several
samples a thread; sums beyond 64 and 96 bits; energies of either sign."""
import pytest

import oracle
from paper_1903_11714_gb300 import build as libbuild
from paper_1903_11714_gb300 import ising

pytestmark = pytest.mark.gpu

# n, N and the sums round once to FP64 and each quotient is two products and a division: eight
# roundings at most, and U4 at most twice that of a ratio below 1.
REL = 8 * 2.0 ** -53
ABS_BINDER = 32 * 2.0 ** -53


@pytest.fixture(scope="module", autouse=True)
def _lib():
    libbuild.build()
    ising.lib()


@pytest.mark.parametrize("L,beta,start", [(64, 1e-3, ising.HOT), (64, 0.44, ising.HOT), (8192, 0.6, ising.COLD)])
def test_moments_at_the_edges_of_the_reduction(L, beta, start):
    last = 4200 if L == 64 else 140
    lat = ising.Lattice(L, beta, 11, start).sweep(last)
    M, E = lat.history()
    for count in (1, 31, 32, 33, 127, 512, 513, 2047, 2048, 2049, 4196):
        if count > last:
            break
        got, ex = lat.moments(last - count), oracle.moments_exact(M, E, L * L, last - count)
        for k in ("S1", "S2", "S4", "SE", "SE2"):
            assert got[k] == ex[k], (count, k)
        for k in ("abs_m", "m2", "m4", "e", "e2"):
            assert got[k] == pytest.approx(ex[k], rel=REL, abs=0), (count, k)
        assert got["binder"] == pytest.approx(ex["binder"], rel=0, abs=ABS_BINDER), count
    lat.close()
