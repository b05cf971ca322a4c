"""First layer of the tensor-core inference reading the FP32 image itself (GPU).

Widths around one strip of 128 pixels (the ghost column in the strip's last slot, in the
next strip's first, alone in a strip), heights around the rows kept in flight and the ring,
and bands with a short last one.  Compared with the FP64 network as in the inference tests.
"""
import numpy as np
import pytest

from tests.test_gpu_cnn_infer import _params, _run, check_against_oracle, oracle_view

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny", [(126, 1), (127, 3), (129, 4), (130, 6), (255, 7), (257, 5), (2, 2), (384, 701)])
def test_image_rows_match_the_oracle(gpu, nx, ny):
    p32 = _params(nx * 3 + ny)
    x = np.random.default_rng(nx + ny).normal(size=(4, ny, nx)).astype(np.float32)
    check_against_oracle(_run(nx, ny, p32, x), oracle_view(p32), x.astype(np.float64))
