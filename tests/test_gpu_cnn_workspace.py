"""A CNN workspace may lie at any address: results at offsets of 1 to 255 bytes are those of
an aligned workspace bit for bit."""
import ctypes as C

import numpy as np
import pytest

from oracle import cnn_oracle as N
from paper_2101_04847_gb300 import lbm

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("offset", [1, 4, 8, 24, 255])
def test_workspace_at_any_address(gpu, offset):
    import torch

    nx, ny = 70, 21
    rng = np.random.default_rng(offset)
    p, x, t = (torch.from_numpy(a.astype(np.float32)).cuda()
               for a in (N.init_params(1), rng.normal(size=(4, ny, nx)), rng.normal(size=(4, ny, nx))))
    n = C.c_size_t()
    assert gpu.lbm_cnn_workspace_bytes(nx, ny, C.byref(n)) == lbm.LBM_OK
    buf = torch.empty(n.value + 512, dtype=torch.uint8, device="cuda")
    stream = C.c_void_p(torch.cuda.current_stream().cuda_stream)
    results = []
    for off in (0, offset):
        buf.fill_(0xff)
        ws = C.c_void_p(buf.data_ptr() + off)
        a, b, grad, loss = torch.empty_like(x), torch.empty_like(x), torch.empty_like(p), C.c_double()
        args = (C.c_void_p(p.data_ptr()), C.c_void_p(x.data_ptr()), nx, ny, ws, n.value, stream)
        assert gpu.lbm_cnn_forward(*args, C.c_void_p(a.data_ptr())) == lbm.LBM_OK
        assert gpu.lbm_cnn_infer(*args, C.c_void_p(b.data_ptr())) == lbm.LBM_OK
        assert gpu.lbm_cnn_infer_status(ws, nx, ny, stream) == lbm.LBM_OK
        assert gpu.lbm_cnn_loss_grad(*args[:2], C.c_void_p(t.data_ptr()), *args[2:], C.byref(loss),
                                     C.c_void_p(grad.data_ptr())) == lbm.LBM_OK
        results.append((loss.value, *(v.cpu().numpy() for v in (a, b, grad))))
        # nothing is written outside the workspace
        assert bool((buf[:off] == 0xff).all()) and bool((buf[off + n.value:] == 0xff).all())
    assert results[0][0] == results[1][0]
    for u, v in zip(results[0][1:], results[1][1:]):
        assert np.array_equal(u, v)
