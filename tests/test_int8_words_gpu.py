"""GPU parity of the byte-per-spin half-sweep at the edges of its two word layouts: 64-byte
segments in strips of 2 to 16 rows (L % 64 == 0), and words of eight 8-byte chunks that
straddle rows (every other multiple of 8)."""
import numpy as np
import pytest

import oracle
from paper_1903_11714_gb300 import build as libbuild
from paper_1903_11714_gb300 import ising

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    libbuild.build()
    ising.lib()


def run(L, beta, seed, sweeps):
    lat = ising.Lattice(L, beta, seed, ising.HOT, ising.INT8).sweep(sweeps)
    out = lat.history(0, sweeps), lat.get_lattice()
    lat.close()
    return out


@pytest.mark.parametrize("L", [8, 16, 24, 40, 56, 64, 72, 120, 128, 192, 200, 1000, 1024])
@pytest.mark.parametrize("beta", [0.0, 0.4406868, 200.0])
def test_matches_oracle(L, beta):
    (M, E), got = run(L, beta, 31 + L, 12)
    ref, m, e, _ = oracle.run(L, beta, 31 + L, oracle.HOT, 12)
    assert np.array_equal(M, m) and np.array_equal(E, e)
    assert np.array_equal(got, ref)


@pytest.mark.parametrize("L", [2048, 4096, 4160, 8192])  # strips of 2, 4, 4 and 16 rows
def test_strips_match_packed(L):
    (M, E), got = run(L, 0.43, 5, 4)
    lat = ising.Lattice(L, 0.43, 5, ising.HOT).sweep(4)
    m, e = lat.history(0, 4)
    assert np.array_equal(M, m) and np.array_equal(E, e)
    assert np.array_equal(got, lat.get_lattice())
    lat.close()
