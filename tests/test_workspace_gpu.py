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
