"""Runs that are too short, or too early, for random numbers drawn ahead: one launch of the resident
kernel (L <= 256) or two a sweep of the tiled one (large lattices), before and after longer runs, and
captured into a graph."""
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


RESIDENT, AHEAD = (ising.RUN_RESIDENT, 1), ising.RUN_AHEAD


def check(lat, L, beta, seed, n):
    ref, M, E, _ = oracle.run(L, beta, seed, ising.HOT, n)
    m, e = lat.history(0, n)
    assert np.array_equal(m, M) and np.array_equal(e, E)
    assert np.array_equal(lat.get_lattice(), ref)


# (run, form): a new handle's first runs, one long enough to take the workspace, then the lengths on
# either side of where a launch to draw and one to update are the faster
@pytest.mark.parametrize("L,runs", [
    (64, [(1, RESIDENT), (15, RESIDENT), (70, RESIDENT), (30, AHEAD), (1, RESIDENT), (3, RESIDENT), (4, AHEAD), (8, AHEAD), (9, AHEAD)]),
    (128, [(1, RESIDENT), (15, RESIDENT), (47, RESIDENT), (20, AHEAD), (1, RESIDENT), (5, RESIDENT), (6, AHEAD)]),
    (192, [(1, RESIDENT), (15, RESIDENT), (40, AHEAD), (2, RESIDENT), (3, AHEAD)]),
    (256, [(1, RESIDENT), (14, RESIDENT), (17, AHEAD), (1, RESIDENT), (2, AHEAD)]),
])
@pytest.mark.parametrize("beta", [0.0, 0.4406868, 200.0])
def test_forms_and_chain(L, runs, beta):
    lat = ising.Lattice(L, beta, 11 + L, ising.HOT)
    for n, form in runs:
        lat.sweep(n)
        assert lat.last_run() == form if form == RESIDENT else lat.last_run()[0] == form
    check(lat, L, beta, 11 + L, sum(n for n, _ in runs))
    lat.close()


@pytest.mark.parametrize("L", [64, 128, 192, 256])
def test_captured_at_once(L):
    # a program that captures its run right after it made the handle
    import torch

    stream = torch.cuda.Stream()
    lat = ising.Lattice(L, 0.43, 32, ising.HOT, stream=stream)
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=stream, capture_error_mode="thread_local"):
        lat.sweep(100)
    assert lat.last_run() == RESIDENT
    with torch.cuda.stream(stream):
        g.replay()
    check(lat, L, 0.43, 32, 100)
    del g
    lat.close()


@pytest.mark.parametrize("L,runs", [(5504, [(20, AHEAD), (1, AHEAD), (2, AHEAD)]),
                                    (5568, [(20, AHEAD), (1, ising.RUN_TILED), (2, AHEAD)]),
                                    (8192, [(20, AHEAD), (1, ising.RUN_TILED), (2, ising.RUN_TILED), (3, AHEAD)])])
def test_one_or_two_sweeps_of_large_lattices(L, runs):
    lat = ising.Lattice(L, 0.43, 6, ising.HOT)
    n = sum(r for r, _ in runs)
    for r, form in runs:
        lat.sweep(r)
        assert lat.last_run()[0] == form
    b = ising.Batch(1, L, L * L // 8 + 16 * n + 4096)
    b.set_cluster(ising.CLUSTER_OFF)
    k = b.add(L, 0.43, 6, ising.HOT, n)
    b.run(n)
    assert all(np.array_equal(x, y) for x, y in zip(lat.history(0, n), b.history(k)))
    assert np.array_equal(lat.get_lattice(), b.get_lattice(k))
    lat.close()
    b.close()


# batches: one sweep, two from 5e6 sites on, three from 3e7 and four from 8e7 on go to the kernels that draw as they go
@pytest.mark.parametrize("Ls,shortest", [([64, 320, 512], 2), ([2048, 1024, 512, 64], 3), ([4096, 4096], 4), ([4096] * 5, 5)])
@pytest.mark.parametrize("graph", [False, True])
def test_short_batch_runs(Ls, shortest, graph):
    runs, out = [35, 1, 2, 3, 4, 5], []
    for mode in (ising.CLUSTER_AUTO, ising.CLUSTER_OFF):
        b = ising.Batch(len(Ls), max(Ls), sum(L * L // 8 + 16 * 50 + 4096 for L in Ls) + (1 << 25))
        b.set_cluster(mode)
        idx = [b.add(L, 0.35 + 0.05 * k, 70 + k, ising.HOT, 50) for k, L in enumerate(Ls)]
        for n in runs:
            b.run(n, n if graph else 0)
            assert (b.last_run()[0] == ising.RUN_AHEAD) == (mode == ising.CLUSTER_AUTO and n >= shortest)
        out.append([(*b.history(i), b.get_lattice(i)) for i in idx])
        b.close()
    for short, tiled in zip(*out):
        assert all(np.array_equal(a, t) for a, t in zip(short, tiled))
