"""CPU: rules of the kernels' source that no run can show, because a program that breaks one
may still work as compiled."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1312_2415_gb300", "csrc")


def code(path):
    text = re.sub(r"/\*.*?\*/", "", open(path).read(), flags=re.S)
    return re.sub(r"//[^\n]*", "", text)


def test_warp_barriers_name_their_lanes():
    """The active mask says which lanes happen to be together, not which have to meet: a
    barrier or exchange over it orders nothing between lanes that diverged before it."""
    files = sorted(glob.glob(os.path.join(CSRC, "*.cu")))
    assert files
    for f in files:
        assert "__activemask" not in code(f), f
