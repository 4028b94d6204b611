"""Batches and lattices that the estimates give to the drawn-ahead form take it, and their chain is the
tiled kernel's: each side's form is asserted, so that neither is compared with itself."""
import numpy as np
import pytest

from paper_1903_11714_gb300 import build as libbuild
from paper_1903_11714_gb300 import ising

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    libbuild.build()
    ising.lib()


# one-tile lattices only; every strip height; long rows; tall tiles (2e6 sites and more); several of one
# side, which a cluster could hold
@pytest.mark.parametrize("Ls", [[64, 128, 192], [64, 128, 192, 256, 320, 384, 448, 512, 1088], [4096, 64, 2112],
                                [2048, 960, 1536, 1344], [3072, 1024, 128, 640], [1024] * 4])
def test_batch_forms(Ls):
    out = []
    for mode in (ising.CLUSTER_AUTO, ising.CLUSTER_OFF):
        b = ising.Batch(len(Ls), max(Ls), sum(L * L // 8 + 16 * 100 + 4096 for L in Ls) + (1 << 25))
        b.set_cluster(mode)
        idx = [b.add(L, 0.3 + 0.05 * (k % 7), 50 + k, ising.HOT, 100) for k, L in enumerate(Ls)]
        b.run(40)
        forms = [b.last_run()[0]]
        b.run(11)
        forms.append(b.last_run()[0])
        assert forms == [ising.RUN_AHEAD if mode == ising.CLUSTER_AUTO else ising.RUN_TILED] * 2
        out.append([(*b.history(i), b.get_lattice(i)) for i in idx])
        b.close()
    for ahead, tiled in zip(*out):
        assert all(np.array_equal(a, t) for a, t in zip(ahead, tiled))


@pytest.mark.parametrize("L", [64, 128, 192, 256, 320, 512, 1024, 4160, 8192])
def test_single_forms(L):
    lat = ising.Lattice(L, 0.43, 9, ising.HOT).sweep(100)
    assert lat.last_run()[0] == ising.RUN_AHEAD
    b = ising.Batch(1, L, L * L // 8 + 16 * 100 + 4096)
    b.set_cluster(ising.CLUSTER_OFF)
    k = b.add(L, 0.43, 9, ising.HOT, 100)
    b.run(100)
    assert b.last_run()[0] == ising.RUN_TILED
    assert all(np.array_equal(a, t) for a, t in zip(lat.history(0, 100), b.history(k)))
    assert np.array_equal(lat.get_lattice(), b.get_lattice(k))
    lat.close()
    b.close()
