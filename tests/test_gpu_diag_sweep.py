"""The diagnostics sweep at the edges of its tiles: grids narrower than its halo, one
column more or less than a block's, averaged rows that begin or end beside a tile's edge,
few averaged rows, row batches that are not full.  Tolerances as in
test_gpu_diagnostics: 1e-9 of the largest budget term."""
import numpy as np
import pytest

from oracle import lbm_oracle as O
from paper_2101_04847_gb300 import lbm
from tests import inputs
from tests.test_gpu_diagnostics import check_diag, evolved_state

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,crop,storage", [(4, 8, 3, "f32"), (5, 40, 12, "f32"), (124, 33, 4, "f32"),
                                                (125, 64, 31, "f32"), (249, 65, 3, "f32"), (123, 47, 5, "f32"),
                                                (60, 41, 7, "f16"), (125, 36, 3, "bf16")])
def test_diagnostics_at_tile_edges(gpu, nx, ny, crop, storage):
    d = inputs.params(inputs.C0, nx=nx, ny=ny, g=1e-4, amp=min(2.0, ny / 16), crop_rows=crop, wall_mode=nx % 2)
    f, p = evolved_state(d, 30)
    with lbm.Solver(storage=storage, **d) as s:
        s.set_populations(f)
        state = s.populations()   # the state as stored
        got = s.diagnostics()
        rows = s.profile()
    ref = O.diagnostics(state, p)
    check_diag(got, ref)
    assert np.max(np.abs(rows - ref["phi_rows"])) <= 1e-12
