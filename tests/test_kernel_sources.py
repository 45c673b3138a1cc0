"""Rules that the CUDA sources keep and that no run of today's build can show."""

import pathlib
import re

CSRC = pathlib.Path(__file__).resolve().parent.parent / "paper_2109_03592_gb300" / "csrc"


def _code(path):
    return re.sub(r"//[^\n]*", "", path.read_text())


def test_warp_operations_name_their_lanes():
    """__activemask() returns whichever lanes happen to be converged: as the mask of a warp operation behind a branch it
    can leave lanes with values of their own out."""
    for path in sorted(CSRC.glob("*.cu*")):
        assert "__activemask" not in _code(path), path.name
