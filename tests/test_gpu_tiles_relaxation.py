"""With relaxation times other than 1 no product of the collision is exact: the states still
do not depend on the step kernel, the tile shape or the ensemble, bit for bit."""
import numpy as np
import pytest

from paper_2101_04847_gb300 import lbm
from tests import inputs

pytestmark = pytest.mark.gpu

SHAPES = [dict(tile_x=128, tile_y=5), dict(tile_x=256, tile_y=16), dict(kernel="decoupled"), dict(kernel="fused"),
          dict(kernel="warp"), dict(kernel="two_pass")]


@pytest.mark.parametrize("storage", ["f32", "f16", "bf16"])
@pytest.mark.parametrize("nx,ny", [(33, 21), (257, 90)])
def test_states_do_not_depend_on_the_tiles(gpu, storage, nx, ny):
    d = inputs.params(inputs.C0, nx=nx, ny=ny, crop_rows=3, g=1e-4, tau_A=0.7, tau_B=1.3, storage=storage,
                      amp=min(2.0, ny / 16))
    f = inputs.random_populations(nx, nx, ny).astype(np.float32)

    def run(solver):
        solver.set_populations(f)
        solver.step(5)
        return solver.populations()

    with lbm.Solver(**d) as s:
        want = run(s)
    same_arithmetic = SHAPES if storage == "f32" else SHAPES[:3]   # the others form f = h + w rho0 first
    for shape in same_arithmetic:
        with lbm.Solver(**dict(d, **shape)) as s:
            assert np.array_equal(run(s), want), shape
    for tile in (dict(), dict(tile_y=7, tile_x=128)):
        with lbm.Ensemble([lbm.default_params(**d, **tile) for _ in range(2)]) as e:
            for m in e.members:
                m.set_populations(f)
            e.step(5)
            for m in e.members:
                assert np.array_equal(m.populations(), want), tile
