"""Shuffle masks name the lanes that take part (CPU, from the sources): the set of lanes that
happen to be active at an instruction is not one that the programming model promises."""
import glob
import os

CSRC = os.path.join(os.path.dirname(__file__), "..", "paper_2607_12201_gb300", "csrc")


def test_no_mask_from_the_active_lanes():
    files = glob.glob(os.path.join(CSRC, "*.cu*"))
    assert files
    assert not [f for f in files if "__activemask" in open(f).read()]
