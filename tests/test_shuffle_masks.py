"""Shuffle masks in the kernels: never __activemask, which reports the lanes that
happen to be converged, not those that take part."""
import glob
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_no_mask_from_the_lanes_that_happen_to_be_converged():
    files = glob.glob(os.path.join(ROOT, "paper_2607_24908_gb300", "csrc", "*.cu*"))
    assert files
    for name in files:
        with open(name) as f:
            assert "__activemask" not in re.sub(r"//[^\n]*", "", f.read()), name
