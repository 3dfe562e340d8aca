"""The checked build tests every index that comes from data: in the render
kernels' source, each access to a buffer of the near pass goes through
GBRT_INDEX (the GPU tests of the checked build then run them)."""
import os
import re

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_0801_1500_gb300", "csrc",
                   "render.cu")


def test_near_pass_buffers_are_indexed_through_the_check():
    src = open(SRC).read()
    found = re.findall(r"\bb\.(tiles|units|masks)\[(\w+)", src)
    assert {k for k, _ in found} == {"tiles", "units", "masks"}
    assert all(i == "GBRT_INDEX" for _, i in found), found
    found = re.findall(r"grid\.(bstart|balls) \+ (\w+)", src)
    assert {k for k, _ in found} == {"bstart", "balls"}
    assert all(i == "GBRT_INDEX" for _, i in found), found
