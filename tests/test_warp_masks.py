"""Warp-wide operations of the CUDA sources name the lanes that take part: __activemask() reports whichever
lanes happen to be together, which after a branch need not be the warp, so no mask is made from it."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2603_14641_gb300", "csrc")


def test_no_mask_from_convergence():
    found = []
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        code = re.sub(r"//[^\n]*|/\*.*?\*/", "", open(path).read(), flags=re.S)
        found += [os.path.basename(path)] * code.count("__activemask")
    assert not found, found
