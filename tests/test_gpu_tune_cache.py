"""Lines of a tuner's cache file that were written for other step kernels (no revision in
their key, or another one) are not used."""
import pytest

from paper_2101_04847_gb300 import lbm
from tests import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("suffix", ["", "|r1"])
def test_lines_of_other_kernels_are_skipped(gpu, tmp_path, suffix):
    import torch

    d = inputs.params(inputs.C0, nx=300, ny=200)
    name = torch.cuda.get_device_name(0).replace(" ", "_")
    stale = f"{name}|{lbm.KERNEL['staged']}|0|300x200{suffix} 128 96 0.000001\n"
    cache = tmp_path / "tune.txt"
    cache.write_text(stale)
    with lbm.Solver(kernel="staged", **d) as s:
        _, ms = s.tune(cache)
    assert ms > 1e-4          # timed, not read
    lines = cache.read_text().splitlines(keepends=True)
    assert lines[0] == stale and len(lines) == 2 and lines[1].startswith(f"{name}|{lbm.KERNEL['staged']}|0|300x200|r")
    with lbm.Solver(kernel="staged", **d) as s:
        assert s.tune(cache)[1] == pytest.approx(ms, rel=1e-3)   # found under its own key
    assert cache.read_text().splitlines(keepends=True) == lines
