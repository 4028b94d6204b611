"""GPU parity of the 3D half-sweep for the word groups of a thread (rows of an even number of words
in pairs, of a multiple of three in threes, others singly) and cubes too small to give every
warp a full turn."""
import numpy as np
import pytest

import oracle
from paper_1903_11714_gb300 import build as libbuild
from paper_1903_11714_gb300 import ising

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L", [192, 256, 320, 384])  # 3, 4, 1 and 2 words a group
@pytest.mark.parametrize("mode", [ising.SPECIALIZE_OFF, ising.SPECIALIZE_ALWAYS])
def test_groups_match_oracle(L, mode):
    libbuild.build()
    ising.ising_set_specialize(mode)
    try:
        lat = ising.Lattice3D(L, 0.22, 3 + L, ising.HOT)
    finally:
        ising.ising_set_specialize(ising.SPECIALIZE_AUTO)
    lat.sweep(2)
    ref, M, E, _ = oracle.run3d((L, L, L), 0.22, 3 + L, oracle.HOT, 2)
    m, e = lat.history(0, 2)
    assert np.array_equal(m, M) and np.array_equal(e, E)
    assert np.array_equal(lat.get_lattice(), ref)
    lat.close()
