"""Rules that every kernel source keeps and that no run can show."""
import os

import pytest

CSRC = os.path.join(os.path.dirname(os.path.abspath(__file__)), os.pardir, "paper_1712_06121_gb300", "csrc")
SOURCES = sorted(f for f in os.listdir(CSRC) if f.endswith((".cu", ".cuh", ".h")))


def _code(name):
    """The source's lines without // comments."""
    with open(os.path.join(CSRC, name)) as f:
        return "\n".join(line.split("//")[0] for line in f)


# the lanes that happen to be converged are not a set that a warp may be told
# to work as: a mask follows from indices or from a vote of the whole warp
@pytest.mark.parametrize("name", SOURCES)
def test_warp_masks_do_not_rest_on_convergence(name):
    assert "__activemask" not in _code(name)
