"""The layouts that outlive the stored one: state files hold planes of one component
and direction, [component][direction][ny][pitch] values with column 0 128 bytes into a
row and periodic ghost columns, whatever the layout in device memory is."""
import ctypes as C

import numpy as np
import pytest

from paper_2101_04847_gb300 import lbm
from tests import inputs

pytestmark = pytest.mark.gpu

CX = (0, 1, 0, -1, 0, 1, -1, -1, 1)
CY = (0, 0, 1, 0, -1, 1, 1, -1, -1)
OPP = (0, 3, 4, 1, 2, 7, 8, 5, 6)


@pytest.mark.parametrize("storage,dtype", [("f32", np.float32), ("f16", np.float16)])
@pytest.mark.parametrize("nx,ny", [(4, 8), (131, 21), (256, 16)])
def test_state_file_planes(gpu, tmp_path, storage, dtype, nx, ny):
    d = inputs.params(inputs.C0, nx=nx, ny=ny, crop_rows=3, storage=storage, seed=5)
    path = tmp_path / "state.bin"
    with lbm.Solver(**d) as s:
        s.step(7)
        s.save(path)
        want = s.populations()
    raw = path.read_bytes()
    head = np.frombuffer(raw[8:32], dtype=np.int32)
    assert raw[:8] == b"LBMSTAT1" and list(head[:3]) == [1, nx, ny]
    pitch, size = int(head[4]), np.dtype(dtype).itemsize
    origin = 128 // size
    assert pitch == (origin + max(nx + 160, -(-nx // 256) * 256 + 8) + 63) // 64 * 64
    planes = np.frombuffer(raw[48 + C.sizeof(lbm.LbmParams):], dtype=dtype).reshape(2, 9, ny, pitch)
    assert np.array_equal(planes[..., origin - 2:origin], planes[..., origin + nx - 2:origin + nx])
    assert np.array_equal(planes[..., origin + nx:origin + nx + 2], planes[..., origin:origin + 2])
    b = planes[..., origin:origin + nx].astype(np.float64)
    if storage == "f16":   # h = f - w_i rho0_s, in FP32 as the library forms it
        w = np.array([4 / 9] + [1 / 9] * 4 + [1 / 36] * 4, dtype=np.float32).astype(np.float64)
        shift = np.array([0.5 * m * (1 + d["minority"]) for m in (d["mass_A"], d["mass_B"])], dtype=np.float32)
        b = (b + w[None, :, None, None] * shift.astype(np.float64)[:, None, None, None]).astype(np.float32).astype(np.float64)
    got = np.empty_like(b)
    for i in range(9):
        m = np.roll(b[:, i], CX[i], axis=-1)
        for y in range(ny):
            src = y - CY[i]
            got[:, i, y] = m[:, src] if 0 <= src < ny else b[:, OPP[i], y]
    assert np.array_equal(got, want)
    with lbm.Solver(**d) as s:
        s.load(path)
        assert np.array_equal(s.populations(), want)
