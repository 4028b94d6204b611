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


# runs of one handle that alternate between the launch that draws its own masks, the tiled kernel
# (until 16 sweeps have been asked for) and the masks drawn ahead
@pytest.mark.parametrize("L,runs", [(64, [1, 9, 2, 3, 8, 1, 20]), (128, [2, 3, 1, 5, 2, 9, 1]), (256, [1, 9, 3, 5, 1])])
def test_routes_alternate(L, runs):
    lat = ising.Lattice(L, 0.43, 31, ising.HOT)
    check(lat, L, 0.43, 31, ising.HOT, runs)
    lat.close()


# a run captured into a caller's graph, before (9 sweeps) and after (20) the workspace exists
@pytest.mark.parametrize("L", [64, 192, 512])
@pytest.mark.parametrize("before", [9, 20])
def test_captured_run(L, before):
    import torch

    stream = torch.cuda.Stream()
    lat = ising.Lattice(L, 0.43, 32, ising.HOT, stream=stream)
    lat.sweep(before)
    lat.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=stream, capture_error_mode="thread_local"):
        lat.sweep(17)
    with torch.cuda.stream(stream):
        g.replay()
    lat.sweep(4)
    ref, M, E, _ = oracle.run(L, 0.43, 32, ising.HOT, before + 21)
    m, e = lat.history(0, before + 21)
    assert np.array_equal(m, M) and np.array_equal(e, E)
    assert np.array_equal(lat.get_lattice(), ref)
    del g
    lat.close()


def test_captured_batch_run_follows_the_batch():
    # a graph of a batch's run, replayed after another lattice has joined, sweeps it too
    import torch

    stream = torch.cuda.Stream()
    b = ising.Batch(4, 320, 1 << 22, 0, stream)
    first = b.add(320, 0.41, 7, ising.HOT, 100)
    b.add(64, 0.39, 9, ising.HOT, 100)
    b.run(20)
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=stream, capture_error_mode="thread_local"):
        b.run(17)
    second = b.add(128, 0.44, 8, ising.HOT, 100)
    with torch.cuda.stream(stream):
        g.replay()
    b.run(5)
    for k, L, beta, seed, n in ((first, 320, 0.41, 7, 42), (second, 128, 0.44, 8, 22)):
        ref, M, E, _ = oracle.run(L, beta, seed, ising.HOT, n)
        m, e = b.history(k)
        assert np.array_equal(m, M) and np.array_equal(e, E)
        assert np.array_equal(b.get_lattice(k), ref)
    del g
    b.close()


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


def batch_of(Ls, limits, mode=ising.CLUSTER_AUTO):
    b = ising.Batch(len(Ls) + 2, max(Ls), sum(L * L // 8 + 16 * n + 4096 for L, n in zip(Ls, limits)) + (1 << 22))
    b.set_cluster(mode)
    betas = [0.3 + 0.05 * (k % 7) for k in range(len(Ls))]
    idx = [b.add(L, be, 50 + k, ising.HOT if k % 2 else ising.COLD, n)
           for k, (L, be, n) in enumerate(zip(Ls, betas, limits))]
    return b, betas, idx


def test_batch_matches_oracle():
    # one-tile lattices (strips of 2 and 4 rows) and lattices of several tiles; limits inside a
    # chunk, at its end and beyond the runs; runs shorter and longer than a chunk of 16 sweeps
    Ls = [64, 128, 192, 256, 320, 384, 448, 512, 1088]
    limits = [200, 16, 33, 200, 47, 48, 200, 20, 200]
    b, betas, idx = batch_of(Ls, limits)
    for n in (16, 5, 32, 1):
        b.run(n)
    for k, L in enumerate(Ls):
        done = min(limits[k], 54)
        ref, M, E, _ = oracle.run(L, betas[k], 50 + k, ising.HOT if k % 2 else ising.COLD, done)
        m, e = b.history(idx[k])
        assert b.sweeps_done(idx[k]) == done
        assert np.array_equal(m, M) and np.array_equal(e, E), L
        assert np.array_equal(b.get_lattice(idx[k]), ref), L
    b.close()


@pytest.mark.parametrize("Ls", [[4096, 64, 2112], [2048, 960, 1536, 1344], [3072, 1024, 128, 640]])
def test_batch_matches_tiled(Ls):
    out = []
    for mode in (ising.CLUSTER_AUTO, ising.CLUSTER_OFF):
        b, _, idx = batch_of(Ls, [60] * len(Ls), mode)
        for n in (20, 7):
            b.run(n)
        # a lattice leaves and another joins between runs (its slot and places are reused)
        b.remove(idx[1])
        new = b.add(320, 0.41, 99, ising.HOT, 60)
        b.run(17)
        out.append([(b.history(i), b.get_lattice(i)) for i in (idx[0], idx[2], new)])
        b.close()
    for ((ma, ea), la), ((mt, et), lt) in zip(*out):
        assert np.array_equal(ma, mt) and np.array_equal(ea, et) and np.array_equal(la, lt)


# L = 64 in one tile (chunks of 64 and 128 sweeps), L = 128 in tiles of 4 own slices (chunks of 3)
@pytest.mark.parametrize("L,runs", [(64, [20, 70, 150, 1]), (128, [17, 3, 2])])
@pytest.mark.parametrize("beta", [0.0, 0.2216546, 200.0])
def test_cube_matches_oracle(L, runs, beta):
    n = sum(runs)
    lat = ising.Lattice3D(L, beta, 7 + L, ising.HOT)
    for r in runs:
        lat.sweep(r)
    ref, M, E, _ = oracle.run3d((L, L, L), beta, 7 + L, oracle.HOT, n)
    m, e = lat.history(0, n)
    assert np.array_equal(m, M) and np.array_equal(e, E)
    assert np.array_equal(lat.get_lattice(), ref)
    lat.close()
