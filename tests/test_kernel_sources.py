"""Properties of the kernel sources that a run on one machine does not show."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2605_01313_gb300", "csrc")


def code(path):
    """The source without its comments."""
    text = open(path).read()
    return re.sub(r"//[^\n]*|/\*.*?\*/", "", text, flags=re.S)


def test_warp_masks_are_not_taken_from_activity():
    """Which lanes are active after a loop of differing trip counts is up to the
    compiler: a reduction over __activemask() may leave lanes out."""
    sources = sorted(glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.cuh")))
    assert sources
    for path in sources:
        assert "__activemask" not in code(path), os.path.basename(path)
