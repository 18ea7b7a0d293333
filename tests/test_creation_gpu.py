"""Creating a lattice looks at its flags once, in the library: whether a wall moves
is asked of it, not searched for again in the host array (1.5 of 11.5 ms for a 300^3 cavity), and stays what it was at creation when the caller reuses the array."""
import numpy as np
import pytest

from gpu_helpers import ensure_built

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("value,moving", [(None, False), (1, False), (2, True), (3, False)])
def test_moving_walls_are_known_to_the_library(value, moving):
    from paper_1112_0850_gb300.lattice import Lattice
    ensure_built()
    flags = None
    if value is not None:
        flags = np.zeros((5, 6, 7), np.uint8)
        flags[2, 3, 4] = value
    lat = Lattice(7, 6, 5, 0.6, flags=flags)
    assert "has_moving_walls" not in vars(lat)
    if flags is not None:
        flags[:] = 2
    assert lat.has_moving_walls is moving
    lat.close()
