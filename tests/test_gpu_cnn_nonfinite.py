"""Infinities keep their meaning in the training kernels."""
import ctypes as C

import numpy as np
import pytest

from oracle import cnn_oracle as N
from paper_2101_04847_gb300 import lbm

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny", [(40, 24), (600, 500)])   # one tile per partial, several
def test_gradient_of_an_infinite_target(gpu, nx, ny):
    # one output of channel 0 is infinitely far from its target: that channel's bias gradient
    # is an infinite sum of finite terms and one infinity, the other channels' are finite
    import torch

    rng = np.random.default_rng(1)
    x, t = (rng.normal(size=(4, ny, nx)).astype(np.float32) for _ in range(2))
    t[0, ny // 2, nx // 3] = np.inf
    dp, dx, dt = (torch.from_numpy(a).cuda() for a in (N.init_params(2).astype(np.float32), x, t))
    cnn, grad, loss = lbm.Cnn(nx, ny), torch.empty_like(dp), C.c_double()
    stream = C.c_void_p(torch.cuda.current_stream().cuda_stream)
    assert gpu.lbm_cnn_loss_grad(*(C.c_void_p(a.data_ptr()) for a in (dp, dx, dt)), nx, ny, C.c_void_p(cnn.ws.data_ptr()),
                                 cnn.ws.numel(), stream, C.byref(loss), C.c_void_p(grad.data_ptr())) == lbm.LBM_OK
    g = grad.cpu().numpy()
    assert loss.value == np.inf
    assert g[-4] == -np.inf and np.all(np.isfinite(g[-3:]))
    w3 = g[10432:11584].reshape(4, 32, 9)
    assert np.all(np.isfinite(w3[1:])) and not np.any(np.isfinite(w3[0]))


@pytest.mark.parametrize("nx,ny", [(1, 1), (3, 5), (31, 17), (33, 6), (130, 23)])
def test_gradient_beside_a_wall_of_an_input_that_is_not_a_number(gpu, nx, ny):
    # x[1] at one pixel of the last row: the taps that reach it from the rows below are NaN
    # (those pixels exist), the taps that would reach it from beyond the wall, and the other
    # channels' taps, are finite: tiles and four-pixel groups stick out of these images
    import torch

    rng = np.random.default_rng(nx + ny)
    x, t = (rng.normal(size=(4, ny, nx)).astype(np.float32) for _ in range(2))
    x[1, ny - 1, nx // 3] = np.nan
    dp, dx, dt = (torch.from_numpy(a).cuda() for a in (N.init_params(3).astype(np.float32), x, t))
    cnn, grad, loss = lbm.Cnn(nx, ny), torch.empty_like(dp), C.c_double()
    stream = C.c_void_p(torch.cuda.current_stream().cuda_stream)
    assert gpu.lbm_cnn_loss_grad(*(C.c_void_p(a.data_ptr()) for a in (dp, dx, dt)), nx, ny, C.c_void_p(cnn.ws.data_ptr()),
                                 cnn.ws.numel(), stream, C.byref(loss), C.c_void_p(grad.data_ptr())) == lbm.LBM_OK
    g = grad.cpu().numpy()
    bad = ~np.isfinite(g[:1152].reshape(32, 4, 3, 3))
    want = np.zeros_like(bad)
    want[:, 1, 1] = True               # from its own row
    want[:, 1, 2] = ny > 1             # from the row below
    assert np.array_equal(bad, want) and np.all(np.isfinite(g[1152:]))
