"""Properties of the CUDA sources that no run can show to be wrong: an instruction
whose precondition the compiler happens to meet today."""
import glob
import os
import re

from paper_1212_0785_gb300 import build


def test_cluster_barriers_need_no_converged_warp():
    """the .aligned forms of barrier.cluster require that all threads of a warp
    execute the instruction together, which nothing guarantees behind a branch
    that depends on the lane"""
    found = 0
    for path in glob.glob(os.path.join(build.CSRC, "*.cu*")):
        for m in re.finditer(r"barrier\.cluster\.[a-z.]+", open(path).read()):
            found += 1
            assert ".aligned" not in m.group(), (os.path.basename(path), m.group())
    assert found >= 2
