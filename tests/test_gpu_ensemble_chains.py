"""Ensembles whose chains hold several members of one storage type: the kernel's search of
its member table (chains of two and three), grids from a few columns to several tiles wide,
launches of more tiles than the device holds at once, and the default tile height; every
member against the same realisation advanced alone (the same tile code, compiled into another
kernel, so equal up to FMA contraction: one unit in the last place of the storage type, as in
test_gpu_ensemble)."""
import numpy as np
import pytest

from paper_2101_04847_gb300 import lbm
from tests import inputs

pytestmark = pytest.mark.gpu

GRIDS = {"f32": [(256, 128), (97, 200), (150, 66), (1030, 90), (40, 33)],
         "f16": [(160, 64), (300, 90), (129, 50), (513, 37), (8, 40)],
         "bf16": [(700, 20), (64, 64), (257, 31), (90, 120), (5, 24)]}
TOL = {"f32": 1e-6, "f16": 2e-3, "bf16": 1.6e-2}


def params(storage, k, nx, ny, **tile):
    d = inputs.params(inputs.C0, nx=nx, ny=ny, crop_rows=5, g=1e-4, seed=7 + k, amp=min(2.0, ny / 16),
                      G=(1.4, 1.2, 0.0)[k % 3], minority=(0.08, 0.08, 0.0)[k % 3], wall_mode=k % 2)
    return lbm.default_params(kernel="staged", storage=storage, **tile, **d)


@pytest.fixture(scope="module")
def alone(gpu):
    """{(storage, k): populations} of every realisation stepped by a handle of its own."""
    out = {}
    for st, grids in GRIDS.items():
        for k, (nx, ny) in enumerate(grids):
            with lbm.Solver(params(st, k, nx, ny)) as s:
                s.step(53)
                out[st, k] = s.populations()
    return out


@pytest.mark.parametrize("tile", [dict(), dict(tile_y=1), dict(tile_y=7, tile_x=128), dict(tile_y=5, tile_x=256)])
@pytest.mark.parametrize("storages", [("f32",), ("f16",), ("bf16", "f32", "f16")])
def test_members_of_long_chains_equal_solo_runs(gpu, alone, storages, tile):
    keys = [(st, k) for k in range(5) for st in storages]
    with lbm.Ensemble([params(st, k, *GRIDS[st][k], **tile) for st, k in keys]) as ens:
        ens.step(53)                     # one 50-step graph + 3 single launches
        ens.sync()
        got = [m.populations() for m in ens.members]
    for (st, k), g in zip(keys, got):
        want = alone[st, k]
        assert float(np.max(np.abs(g - want)) / np.max(np.abs(want))) < TOL[st], (st, k)


def test_one_row_tiles_beyond_the_resident_blocks(gpu):
    # 3 members of 8 x 300 one-row tiles in one chain, two in the other: 7200 and 4800 blocks
    grid = (1000, 300)
    ps = [params("f32", k, *grid, tile_y=1, tile_x=128) for k in range(5)]
    with lbm.Ensemble(ps) as ens:
        ens.step(3)
        got = [m.populations() for m in ens.members]
    for k, g in enumerate(got):
        with lbm.Solver(params("f32", k, *grid)) as s:
            s.step(3)
            want = s.populations()
        assert float(np.max(np.abs(g - want)) / np.max(np.abs(want))) < TOL["f32"], k
