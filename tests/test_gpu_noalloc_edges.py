"""The no-allocation step at the edges of its tiles: the smallest grid, one column more or
less than a block's 128, more column blocks than the device holds at once, a tall narrow grid;
with the options of the handle step (mirror walls, wall forces, a body force).  Two calls
against two handle steps, within the tolerance of test_zz_no_alloc."""
import ctypes as C

import numpy as np
import pytest

from paper_2101_04847_gb300 import lbm
from tests import inputs

pytestmark = pytest.mark.gpu


def call(lib, p, src, dst, stream):
    return lib.lbm_step_noalloc(C.byref(p), C.c_void_p(src.data_ptr()), C.c_void_p(dst.data_ptr()),
                                C.c_void_p(stream.cuda_stream))


@pytest.mark.parametrize("nx,ny", [(4, 8), (5, 9), (127, 9), (128, 8), (129, 40), (257, 8), (131072, 8), (17, 60000)])
@pytest.mark.parametrize("options", [dict(), dict(wall_mode=1, G_wall_A=0.2, G_wall_B=-0.1, gx=1e-4, gravity_mode=1)])
def test_two_calls_equal_two_handle_steps(gpu, nx, ny, options):
    import torch

    d = inputs.params(inputs.C0, nx=nx, ny=ny, crop_rows=3, g=1e-4, **options)
    f0 = inputs.random_populations(nx + 3 * ny, nx, ny).astype(np.float32)
    with lbm.Solver(kernel="two_pass", **d) as s:
        s.set_populations(f0)
        s.step(2)
        want = s.populations()
    p, stream = lbm.default_params(**d), torch.cuda.current_stream()
    a = torch.from_numpy(f0).cuda()
    b, c = torch.full_like(a, float("nan")), torch.full_like(a, float("nan"))
    assert call(gpu, p, a, b, stream) == lbm.LBM_OK
    assert call(gpu, p, b, c, stream) == lbm.LBM_OK
    got = c.double().cpu().numpy()
    assert float(np.max(np.abs(got - want)) / np.max(np.abs(want))) < 2e-6


def test_calls_on_different_arrays_may_overlap(gpu):
    import torch

    p = lbm.default_params(**inputs.params(inputs.C0, nx=700, ny=600, crop_rows=3, g=1e-4))
    chains = [[torch.from_numpy(inputs.random_populations(k, 700, 600).astype(np.float32)).cuda()] for k in range(2)]
    for c in chains:
        c.append(torch.empty_like(c[0]))
    serial = []
    main = torch.cuda.current_stream()
    for a, b in chains:
        u, v = a.clone(), b.clone()
        for _ in range(20):
            assert call(gpu, p, u, v, main) == lbm.LBM_OK
            u, v = v, u
        serial.append(u.cpu())
    torch.cuda.synchronize()
    streams = [torch.cuda.Stream() for _ in chains]
    for _ in range(20):
        for k, s in enumerate(streams):
            assert call(gpu, p, *chains[k], s) == lbm.LBM_OK
            chains[k].reverse()
    torch.cuda.synchronize()
    for k, want in enumerate(serial):
        assert torch.equal(chains[k][0].cpu(), want)
