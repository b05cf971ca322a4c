"""No kernel takes the lanes that happen to be active as the mask of a warp operation: the
language does not promise that all lanes of a branch are among them."""
from pathlib import Path

CSRC = Path(__file__).resolve().parents[1] / "paper_2101_04847_gb300" / "csrc"


def test_warp_operations_name_their_lanes():
    files = sorted(CSRC.glob("*.cu")) + sorted(CSRC.glob("*.cuh"))
    assert files and not [f.name for f in files if "__activemask" in f.read_text()]
