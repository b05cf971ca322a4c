"""The default tiling: whatever tile shape the size picks (one-row tiles on small
grids, 128-column tiles where they span a 16-bit grid), the states are those of tall
256-column tiles bit for bit, through graph replays and single launches."""
import numpy as np
import pytest

from paper_2101_04847_gb300 import lbm
from tests import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("storage", ["f32", "f16", "bf16"])
@pytest.mark.parametrize("nx,ny", [(4, 8), (128, 9), (129, 40), (257, 700), (1100, 150)])
def test_default_tiles_equal_tall_ones(gpu, storage, nx, ny):
    d = inputs.params(inputs.C0, nx=nx, ny=ny, crop_rows=3, g=1e-4, wall_mode=1, G_wall_A=0.1)
    states = []
    for tile in (dict(), dict(tile_x=256, tile_y=23)):
        with lbm.Solver(storage=storage, **tile, **d) as s:
            s.step(53)
            states.append(s.populations())
    assert np.array_equal(states[0], states[1])
