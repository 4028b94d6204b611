"""GPU parity of the sweep with its random numbers drawn ahead of the update (single packed
lattices of side up to 8,192 on the built-in kernels).

Small sides against the oracle; larger ones against the tiled kernel through a batch,
which the batch tests hold to the oracle.  Run lengths cross the places where the path
changes: the launch that draws its own masks, the first and the largest chunk, and a last
chunk shorter than the others.
"""
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


def check(lat, L, beta, seed, start, runs):
    n = sum(runs)
    ref, M, E, _ = oracle.run(L, beta, seed, start, n)
    for r in runs:
        lat.sweep(r)
    m, e = lat.history(0, n)
    assert np.array_equal(m, M) and np.array_equal(e, E)
    assert np.array_equal(lat.get_lattice(), ref)


# one tile: strips of 2 rows (L = 64, 128) and of 4 (192); several tiles beyond, with strips of
# 2, 4 and 8 rows and rows of an even, odd and prime number of words
@pytest.mark.parametrize("L", [64, 128, 192, 256, 320, 384, 448, 512, 1088])
@pytest.mark.parametrize("beta", [0.0, 0.4406868, 200.0])
def test_ahead_matches_oracle(L, beta):
    lat = ising.Lattice(L, beta, 77 + L, ising.HOT)
    check(lat, L, beta, 77 + L, ising.HOT, [1, 2, 17, 33] if L < 512 else [1, 17])
    lat.close()


def test_long_runs_cross_chunks():
    # L = 128: chunks of 64, 1024 and the rest; L = 256: chunks of 24
    for L, runs in ((128, [3, 1200, 40]), (256, [600, 9])):
        lat = ising.Lattice(L, 0.44, 5, ising.COLD)
        check(lat, L, 0.44, 5, ising.COLD, runs)
        lat.close()


@pytest.mark.parametrize("L", [1024, 1472, 2048, 4096, 4160, 8128, 8192])
def test_ahead_matches_tiled_batch(L):
    runs = [1, 16, 11] if L <= 2048 else [2, 9]
    n = sum(runs)
    lat = ising.Lattice(L, 0.43, 9, ising.HOT)
    for r in runs:
        lat.sweep(r)
    b = ising.Batch(1, L, L * L // 8 + 16 * n + 4096)
    b.set_cluster(ising.CLUSTER_OFF)
    k = b.add(L, 0.43, 9, ising.HOT, n)
    b.run(n)
    m, e = b.history(k)
    M, E = lat.history(0, n)
    assert np.array_equal(m, M) and np.array_equal(e, E)
    assert np.array_equal(lat.get_lattice(), b.get_lattice(k))
    lat.close()
    b.close()


def test_planes_set_between_runs():
    # the copies of the planes that several tiles read follow the handle's planes
    L, rng = 512, np.random.default_rng(3)
    lat = ising.Lattice(L, 0.5, 21, ising.HOT).sweep(5)
    new = (rng.integers(0, 2, size=(L, L)) * 2 - 1).astype(np.int8)
    lat.set_lattice(new)
    lat.sweep(20)
    ref, M, E, _ = oracle.run(L, 0.5, 21, ising.HOT, 20, sweep0=5, state=new)
    m, e = lat.history(5, 20)
    assert np.array_equal(m, M) and np.array_equal(e, E)
    assert np.array_equal(lat.get_lattice(), ref)
    lat.close()
