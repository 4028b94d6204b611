"""Workspaces of random numbers drawn ahead: declined, bounded over the process, tried again."""
import gc

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
    gc.collect()  # handles that earlier tests dropped


def check(lat, L, beta, seed, n):
    ref, M, E, _ = oracle.run(L, beta, seed, ising.HOT, n)
    m, e = lat.history(0, n)
    assert np.array_equal(m, M) and np.array_equal(e, E)
    assert np.array_equal(lat.get_lattice(), ref)


@pytest.mark.parametrize("L,other", [(128, ising.RUN_RESIDENT), (512, ising.RUN_TILED)])
def test_declined(L, other):
    lat = ising.Lattice(L, 0.43, 3, ising.HOT)
    for mode, form in ((ising.WORKSPACE_NONE, other), (ising.WORKSPACE_BESIDE, ising.RUN_AHEAD),
                       (ising.WORKSPACE_NONE, other), (ising.WORKSPACE_BESIDE, ising.RUN_AHEAD)):
        lat.set_workspace(mode)
        lat.sweep(64)
        assert lat.last_run()[0] == form
    check(lat, L, 0.43, 3, 256)
    with pytest.raises(ising.IsingError):
        lat.set_workspace(2)
    lat.close()


def test_given_back_when_declined():
    import torch

    L = 8192
    lat = ising.Lattice(L, 0.43, 3, ising.HOT).sweep(32)
    lat.synchronize()
    with_it = torch.cuda.mem_get_info()[0]
    lat.set_workspace(ising.WORKSPACE_NONE)
    assert torch.cuda.mem_get_info()[0] - with_it > 1.4 * L * L  # 1.5 L^2 bytes of masks and 0.25 L^2 of copies
    lat.close()


def test_many_handles_share_a_bound():
    # 117 MB each: 36 fit the 4 GB of all workspaces, the others sweep without, the same chain
    L, n = 8192, 20
    lats = [ising.Lattice(L, 0.43, 5, ising.HOT).sweep(n) for _ in range(40)]
    forms = [lat.last_run()[0] for lat in lats]
    held = forms.count(ising.RUN_AHEAD)
    assert 20 <= held <= 36 and forms.count(ising.RUN_TILED) == 40 - held
    M, E = lats[0].history(0, n)
    for lat in lats[1:]:
        m, e = lat.history(0, n)
        assert np.array_equal(m, M) and np.array_equal(e, E)
    # room again: a handle that was refused tries anew after 1,024 more sweeps
    late = lats[-1]
    lats[0].close()
    late.sweep(n)
    assert late.last_run()[0] == ising.RUN_TILED
    late.sweep(1024)
    assert late.last_run()[0] == ising.RUN_AHEAD
    for lat in lats:
        lat.close()


def same_chain(b, idx, Ls, sweeps):
    """Every lattice of the batch against the tiled kernel alone."""
    for k, L in zip(idx, Ls):
        t = ising.Batch(1, L, L * L // 8 + 16 * sweeps + 4096)
        t.set_cluster(ising.CLUSTER_OFF)
        i = t.add(L, 0.35 + 0.01 * (L // 64), L, ising.HOT, sweeps)
        t.run(sweeps)
        assert all(np.array_equal(x, y) for x, y in zip(b.history(k), t.history(i)))
        assert np.array_equal(b.get_lattice(k), t.get_lattice(i))
        t.close()


def added(b, L, sweeps):
    return b.add(L, 0.35 + 0.01 * (L // 64), L, ising.HOT, sweeps)


# room beside the lattices for chunks of 16, 8 and 4 sweeps (8.25, 4.25 and 2.25 bytes a site), and for none;
# low and, from 2e6 sites on, tall tiles
@pytest.mark.parametrize("Ls", [[320, 64, 448, 576], [1024, 960, 320, 64]])
@pytest.mark.parametrize("room", [8.3, 4.3, 2.3, 1.0])
def test_workspace_in_the_arena(Ls, room):
    import torch

    sweeps, sites = 60, sum(L * L for L in Ls)
    lattices = sum(L * L // 8 + 16 * sweeps + 256 for L in Ls)
    b = ising.Batch(8, 1024, lattices + int(room * sites) + (1 << 14))
    b.set_workspace(ising.WORKSPACE_ARENA)
    idx = [added(b, L, sweeps) for L in Ls]
    held, free = b.usage()[0], torch.cuda.mem_get_info()[0]
    for n in (37, 5, 18):
        b.run(n)
        assert b.last_run()[0] == (ising.RUN_AHEAD if room > 2 else ising.RUN_TILED)
    assert b.usage()[0] == held  # lattices only
    assert free - torch.cuda.mem_get_info()[0] < 4 << 20  # nothing beside the arena (a kernel's first load aside)
    same_chain(b, idx, Ls, sweeps)
    b.close()


def test_workspace_gives_way_to_lattices():
    sweeps, Ls = 64, [512, 320]
    need = [L * L // 8 + 16 * sweeps for L in (512, 320, 1024)]
    b = ising.Batch(8, 1024, sum(-(-n // 256) * 256 for n in need) + (3 << 20))
    b.set_workspace(ising.WORKSPACE_ARENA)
    idx = [added(b, L, sweeps) for L in Ls]
    b.run(16)
    assert b.last_run()[0] == ising.RUN_AHEAD  # 2.98 MB of the 3.1 MB left
    # the rest of the arena is the workspace's: this lattice takes its room
    idx.append(added(b, 1024, sweeps))
    idx.append(added(b, 1024, sweeps))
    b.run(16)
    with pytest.raises(ising.IsingError) as e:
        for _ in range(40):
            added(b, 1024, 5000)
    assert e.value.code == ising.ISING_EBUSY or e.value.code == ising.ISING_ENOMEM
    b.run(48)
    same_chain(b, idx[:2], Ls, sweeps)
    same_chain(b, idx[2:], [1024, 1024], sweeps)
    b.close()


def test_batch_declines_and_gives_back():
    import torch

    Ls, sweeps = [1024] * 3 + [2048] * 3, 200
    b = ising.Batch(6, 2048, sum(L * L // 8 + 16 * sweeps + 256 for L in Ls))
    idx = [b.add(L, 0.35 + 0.01 * (L // 64), L, ising.HOT, sweeps) for L in Ls]
    for mode, form in ((ising.WORKSPACE_NONE, ising.RUN_TILED), (ising.WORKSPACE_BESIDE, ising.RUN_AHEAD),
                       (ising.WORKSPACE_ARENA, ising.RUN_TILED), (ising.WORKSPACE_BESIDE, ising.RUN_AHEAD),
                       (ising.WORKSPACE_NONE, ising.RUN_TILED)):
        b.synchronize()
        free = torch.cuda.mem_get_info()[0]
        b.set_workspace(mode)
        given = torch.cuda.mem_get_info()[0] - free
        assert (given > 8 * sum(L * L for L in Ls)) == (b.last_run()[0] == ising.RUN_AHEAD)
        b.run(40)
        assert b.last_run()[0] == form
    same_chain(b, idx, Ls, sweeps)
    with pytest.raises(ising.IsingError):
        b.set_workspace(3)
    b.close()


def test_outgrown_workspaces_are_given_back():
    # a batch that grows keeps one workspace, at most half as large again as it needs (two sides, so that
    # no cluster form stands in)
    import torch

    b = ising.Batch(16, 2048, 16 * (2048 * 2048 // 8 + 16 * 800 + 256))
    free = torch.cuda.mem_get_info()[0]
    for k in range(16):
        b.add(2048 if k else 1024, 0.35 + 0.01 * k, k, ising.HOT, 800)
        b.run(40)
        assert k < 1 or b.last_run()[0] == ising.RUN_AHEAD
    b.synchronize()
    sites = 16 * 2048 ** 2
    assert free - torch.cuda.mem_get_info()[0] < 1.5 * 8.25 * sites + (64 << 20)
    b.close()


def test_server_keeps_within_its_budget():
    import torch

    from paper_1903_11714_gb300 import serve
    from paper_1903_11714_gb300.workloads import Request

    reqs = [Request(rid=k, arrival=0.0, L=1024, beta=0.38 + 0.01 * k, seed=k, sweeps=100) for k in range(12)]
    srv = serve.Server(hbm_budget_bytes=1 << 26, slots=12, max_L=1024)
    free = torch.cuda.mem_get_info()[0]
    results, st = srv.serve(reqs, realtime=False)
    assert st.completed == 12 and srv.batch.last_run()[0] == ising.RUN_AHEAD
    assert free - torch.cuda.mem_get_info()[0] < 1 << 25  # 104 MB before
    assert st.max_arena_bytes <= 12 * (1024 * 1024 // 8 + 1600 + 256)
    srv.close()
