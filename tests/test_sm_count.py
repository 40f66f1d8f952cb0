"""Grids and rules that fill the GPU ask the device for its SMs: no source file holds a number of them, but for the one
place that asks and its fallback, and the prototype workspace, whose size may not depend on the device."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1506_07656_gb300", "csrc")


def test_sm_count_is_asked_for():
    found = {}
    for p in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        code = re.sub(r"//[^\n]*", "", open(p).read())
        for m in re.finditer(r"\b(148|152|304|608|1216)\b|cudaDevAttrMultiProcessorCount", code):
            found.setdefault(os.path.basename(p), []).append(m.group(0))
    assert found == {"dm_internal.cuh": ["152", "cudaDevAttrMultiProcessorCount"]}
