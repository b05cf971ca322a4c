"""The gradient of an image with more pixels than 512 for each of the at most 2432 partials,
so that a partial covers more tiles than on smaller ones: against the FP64 oracle, with the
tolerances of test_gpu_closure's gradient check."""
import ctypes as C

import numpy as np
import pytest

from oracle import cnn_oracle as N
from paper_2101_04847_gb300 import lbm
from tests.test_gpu_closure import oracle_view

pytestmark = pytest.mark.gpu


def test_gradient_beyond_the_partials_limit(gpu):
    import torch

    nx, ny = 1301, 1003
    assert nx * ny > 2432 * 512
    rng = np.random.default_rng(7)
    p32 = N.init_params(7).astype(np.float32)
    x, t = (rng.normal(size=(4, ny, nx)).astype(np.float32) for _ in range(2))
    cnn = lbm.Cnn(nx, ny)
    dp, dx, dt = (torch.from_numpy(a).cuda() for a in (p32, x, t))
    grad, loss = torch.full_like(dp, float("nan")), C.c_double()
    stream = C.c_void_p(torch.cuda.current_stream().cuda_stream)
    assert gpu.lbm_cnn_loss_grad(*(C.c_void_p(a.data_ptr()) for a in (dp, dx, dt)), nx, ny, C.c_void_p(cnn.ws.data_ptr()),
                                 cnn.ws.numel(), stream, C.byref(loss), C.c_void_p(grad.data_ptr())) == lbm.LBM_OK
    L, g = N.loss_and_grad(oracle_view(p32), x.astype(np.float64), t.astype(np.float64))
    assert abs(loss.value - L) <= 1e-5 * L
    assert np.max(np.abs(grad.double().cpu().numpy() - g)) <= 1e-4 * np.max(np.abs(g))
