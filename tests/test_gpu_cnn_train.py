"""The training kernels at the edges of their tiles (32 x 16 and 32 x 4 pixels, partials
of several tiles): forward and gradients against the FP64 oracle, with the tolerances of
test_gpu_closure's gradient check."""
import ctypes as C

import numpy as np
import pytest

from oracle import cnn_oracle as N
from paper_2101_04847_gb300 import lbm
from tests.test_gpu_closure import oracle_view

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny", [(1, 1), (3, 5), (31, 17), (32, 16), (33, 4), (70, 66), (300, 190)])
def test_forward_and_gradient_at_tile_edges(gpu, nx, ny):
    import torch

    rng = np.random.default_rng(nx + 100 * ny)
    p32 = N.init_params(nx).astype(np.float32)
    p32[1152:1184] = rng.normal(0.0, 0.1, 32)
    x, t = (rng.normal(size=(4, ny, nx)).astype(np.float32) for _ in range(2))
    cnn = lbm.Cnn(nx, ny)
    dp, dx, dt = (torch.from_numpy(a).cuda() for a in (p32, x, t))
    y, grad, loss = torch.full_like(dx, float("nan")), torch.full_like(dp, float("nan")), C.c_double()
    cnn.forward(dp, dx, y)
    stream = C.c_void_p(torch.cuda.current_stream().cuda_stream)
    assert gpu.lbm_cnn_loss_grad(*(C.c_void_p(a.data_ptr()) for a in (dp, dx, dt)), nx, ny, C.c_void_p(cnn.ws.data_ptr()),
                                 cnn.ws.numel(), stream, C.byref(loss), C.c_void_p(grad.data_ptr())) == lbm.LBM_OK
    q = oracle_view(p32)
    ref = N.forward(q, x.astype(np.float64))["y"].numpy()
    assert np.max(np.abs(y.double().cpu().numpy() - ref)) <= 1e-5 * np.max(np.abs(ref))
    L, g = N.loss_and_grad(q, x.astype(np.float64), t.astype(np.float64))
    assert abs(loss.value - L) <= 1e-5 * L
    assert np.max(np.abs(grad.double().cpu().numpy() - g)) <= 1e-4 * np.max(np.abs(g))
