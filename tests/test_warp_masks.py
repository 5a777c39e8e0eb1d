"""Warp-wide operations of the kernels name the lanes that take part, never
``__activemask()``: that is whichever lanes happen to be together, so lanes of
one group could vote in different sets, take different copies of a loop body
and wait for each other's shuffles at different instructions.
"""
import glob
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_no_warp_operation_over_the_active_mask():
    files = glob.glob(os.path.join(ROOT, "paper_2011_13579_gb300", "csrc", "*.cu*"))
    assert files
    for path in files:
        code = re.sub(r"//[^\n]*", "", open(path).read())
        assert "__activemask" not in code, os.path.basename(path)
