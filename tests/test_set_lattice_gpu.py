"""ising_set_lattice: every entry is looked at (the check goes in blocks of 4,096), and the staging
buffer kept between calls serves reads and writes of any size."""
import numpy as np
import pytest

from paper_1903_11714_gb300 import build as libbuild
from paper_1903_11714_gb300 import ising

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    libbuild.build()
    ising.lib()


@pytest.mark.parametrize("kernel,L", [(ising.PACKED, 128), (ising.INT8, 72)])
def test_every_entry_is_checked(kernel, L):
    lat = ising.Lattice(L, 0.4, 1, ising.HOT, kernel)
    before = lat.get_lattice()
    for at in (0, 1, 4095, 4096, L * L - 1):
        for value in (0, 2, -2, 3, -3, 127, -128):
            bad = np.ones(L * L, dtype=np.int8)
            bad[at] = value
            with pytest.raises(ising.IsingError):
                lat.set_lattice(bad.reshape(L, L))
    assert np.array_equal(lat.get_lattice(), before)
    lat.close()


def test_reads_and_writes_share_the_buffer():
    L, rng = 512, np.random.default_rng(4)
    lat = ising.Lattice(L, 0.4, 1, ising.HOT)
    lat.get_rows(3, 2)  # a small buffer first
    for _ in range(3):
        new = (rng.integers(0, 2, size=(L, L)) * 2 - 1).astype(np.int8)
        lat.set_lattice(new)
        assert np.array_equal(lat.get_rows(5, 70), new[5:75])
        assert np.array_equal(lat.get_lattice(), new)
    lat.close()
