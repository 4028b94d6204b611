"""ising_last_run and ising_batch_last_run: the form of the last run and the kernels it enqueued,
against the counts that its schedule makes."""
import pytest

from paper_1903_11714_gb300 import build as libbuild
from paper_1903_11714_gb300 import ising

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    libbuild.build()
    ising.lib()


# chunks of 28 sweeps at L = 512 and of 3 at 8,192, and one launch more, which draws the first
@pytest.mark.parametrize("L,n,launches", [(512, 100, 5), (512, 28, 2), (8192, 30, 11), (8192, 31, 12)])
def test_drawn_ahead(L, n, launches):
    lat = ising.Lattice(L, 0.44, 3, ising.HOT)
    assert lat.last_run() == (ising.RUN_NONE, 0)
    lat.sweep(4)
    assert lat.last_run() == (ising.RUN_TILED, 9)  # two a sweep and the counter's
    lat.sweep(n)
    assert lat.last_run() == (ising.RUN_AHEAD, launches)
    lat.sweep(0)
    assert lat.last_run() == (ising.RUN_AHEAD, launches)
    lat.close()


def test_one_launch_per_half_sweep():
    for make, form, launches in ((lambda: ising.Lattice(128, 0.44, 3, ising.HOT, ising.INT8), ising.RUN_BYTES, 40),
                                 (lambda: ising.Lattice3D(256, 0.22, 3), ising.RUN_CUBIC, 40),
                                 (lambda: ising.Lattice(8256, 0.44, 3), ising.RUN_TILED, 41)):
        lat = make().sweep(20)
        assert lat.last_run() == (form, launches)
        lat.close()


def test_batches():
    b = ising.Batch(4, 1024, 1 << 22)
    for k in range(3):
        b.add(1024, 0.40 + 0.02 * k, k, ising.HOT, 100)
    assert b.last_run() == (ising.RUN_NONE, 0)
    b.set_cluster(ising.CLUSTER_OFF)
    b.run(20)
    assert b.last_run() == (ising.RUN_TILED, 41)
    b.run(20, graph_sweeps=10)
    assert b.last_run() == (ising.RUN_TILED, 42)
    b.set_cluster(ising.CLUSTER_ALWAYS)
    b.run(20)
    assert b.last_run() == (ising.RUN_CLUSTER, 2)
    b.set_cluster(ising.CLUSTER_AUTO)
    b.run(20)
    assert b.last_run() == (ising.RUN_AHEAD, 4)  # chunks of 16: one that draws, two that update, the counters
    b.close()


def test_null_handles():
    assert ising.lib().ising_last_run(None, None, None) == ising.ISING_EINVAL
    assert ising.lib().ising_batch_last_run(None, None, None) == ising.ISING_EINVAL
