"""(M, E) of the byte-per-spin half-sweep where the last warp of strips has fewer than 32: lanes
without a strip of their own still finish words of the warp's queue, and what they finish counts."""
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


# L / 64 odd: strips of 4 rows (16 lanes of the last warp have one), of 8 (8 lanes), of 16 (4 lanes); 8,064:
# strips of 16, L / 64 twice an odd number (16 lanes)
@pytest.mark.parametrize("L", [4032, 5696, 8000, 8064, 8128])
@pytest.mark.parametrize("beta,start", [(0.4406868, ising.HOT), (0.3, ising.HOT), (0.6, ising.COLD)])
def test_last_warp_counts(L, beta, start):
    sweeps = 40
    out = []
    for kernel in (ising.INT8, ising.PACKED):
        lat = ising.Lattice(L, beta, 5, start, kernel).sweep(sweeps)
        out.append((*lat.history(0, sweeps), lat.get_lattice()))
        lat.close()
    (M, E, got), (m, e, ref) = out
    assert np.array_equal(got, ref)
    assert np.array_equal(M, m) and np.array_equal(E, e)


# sides that are no multiple of 64: one word a thread, in blocks of 64 and, from 128 words an SM on, of 128
# threads; whole blocks and a last one with a few words
@pytest.mark.parametrize("L", [8, 88, 200, 488, 1080, 1096, 1112, 1128])
def test_word_blocks(L):
    lat = ising.Lattice(L, 0.42, L, ising.HOT, ising.INT8).sweep(12)
    ref, M, E, _ = oracle.run(L, 0.42, L, oracle.HOT, 12)
    m, e = lat.history(0, 12)
    assert np.array_equal(m, M) and np.array_equal(e, E)
    assert np.array_equal(lat.get_lattice(), ref)
    lat.close()
