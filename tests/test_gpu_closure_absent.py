"""A correction leaves an absent component alone, even where the network's velocity
correction is not finite."""
import numpy as np
import pytest

from oracle import lbm_oracle as O
from paper_2101_04847_gb300 import lbm

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode", [1, 2, 3, 4])
def test_absent_component_keeps_its_populations(gpu, mode):
    with lbm.Closure(lbm.default_params(nx=160, ny=64, mass_B=1.0, crop_rows=10), interval=10, seed=0) as c:
        _, co = c.solvers()
        f = np.repeat(np.repeat(np.outer([1.0, 0.5], O.W)[:, :, None, None], co.ny, axis=2), co.nx, axis=3).astype(np.float32)
        f[1, :, :, co.nx // 2:] = 0.0            # no B on the right
        f[0, :, 3:9, 2:5] = 0.0                  # no A in a patch
        p = np.zeros(lbm.CNN_PARAMS, dtype=np.float32)
        p[-2] = np.inf                           # the output bias of the x velocity
        c.set_params(p)
        c.set_normalisation(np.zeros(4), np.ones(4), np.full(4, 1e-3))
        co.set_populations(f)
        before = co.populations()
        c.correct(mode)
        after = co.populations()
    absent = before.sum(axis=1) == 0.0
    assert absent.any(axis=(1, 2)).all()
    for s in range(2):
        assert np.all(after[s][:, absent[s]] == 0.0), s
    assert not np.all(np.isfinite(after))        # the correction itself did not stay finite
