"""A warp-level synchronisation orders the lanes that its mask names.  `__activemask()` names
the lanes that happen to run together, so a partner lane may be missing from it and its read
be overtaken by a neighbour's write: no kernel synchronises, votes or shuffles on it."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1903_00548_gb300", "csrc")


@pytest.mark.parametrize("name", sorted(f for f in os.listdir(CSRC) if f.endswith((".cu", ".cuh"))))
def test_no_sync_on_the_converged_lanes(name):
    with open(os.path.join(CSRC, name)) as f:
        code = re.sub(r"//[^\n]*", "", f.read())
    assert "__activemask" not in code
