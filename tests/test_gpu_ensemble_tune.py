"""lbm_ens_tune leaves no ensemble slower than it found it: small grids, whose default tiles
have fewer rows than the tuner's candidates, and larger ones."""
import numpy as np
import pytest

from paper_2101_04847_gb300 import lbm
from tests import inputs

pytestmark = pytest.mark.gpu


def us_per_step(ens, steps):
    """The fastest of five runs of 50-step graphs."""
    import torch

    ens.step(steps)
    a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
    out = []
    for _ in range(5):
        a.record()
        ens.step(steps)
        b.record()
        b.synchronize()
        out.append(1e3 * a.elapsed_time(b) / steps)
    return min(out)


# Runs of one side differ by under 2 % (eight 128x256 members 9.87 to 9.93 us a step);
# twice that and what one millisecond's timing inside the tuner can be off are allowed: 10 %.
# Tiles of 12 rows, the tuner's shortest, take 1.6 to 2.6 times as long as the default on the
# first two.
@pytest.mark.parametrize("grids,steps", [([(128, 256, "f32")] * 8, 200),
                                         ([(256, 128, "f32"), (97, 200, "f32"), (160, 64, "f16")], 200),
                                         ([(512, 1024, "f32"), (512, 1024, "f16"), (1024, 512, "f32")], 100)])
def test_tuning_never_slows_an_ensemble(gpu, grids, steps):
    import torch

    params = [lbm.default_params(**inputs.params(inputs.C0, nx=nx, ny=ny, crop_rows=5, storage=st, seed=3 + k))
              for k, (nx, ny, st) in enumerate(grids)]
    with torch.cuda.stream(torch.cuda.Stream()), lbm.Ensemble(params) as ens:
        before = us_per_step(ens, steps)
        state = [m.populations() for m in ens.members]
        _, ms = ens.tune()
        for m, f in zip(ens.members, state):
            assert np.array_equal(m.populations(), f)
        after = us_per_step(ens, steps)
        assert ms > 0 and after <= 1.1 * before, (before, after)
