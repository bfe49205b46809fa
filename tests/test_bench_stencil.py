"""The bench's account of a stencil step: its launches and their names follow the
path that the plan takes (CPU only)."""
import os
import re

import bench

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_launches_follow_the_path():
    src = open(os.path.join(ROOT, "paper_1908_06649_gb300", "csrc", "grid_plan.cu")).read()
    line = int(re.search(r"constexpr int kClosedSteps = (\d+);", src).group(1))
    real, n, text = bench.stencil_launches(3, 16, 256, line)
    assert (real, n) == (True, 4) and "weights" not in text and "extract" not in text
    real, n, text = bench.stencil_launches(3, 16, 256, line + 1)
    assert (real, n) == (True, 12) and "weights" in text and "scattered" in text
    # single products, and tiles beyond one pass per axis: complex tiles
    for args in ((1, 16, 256, 4), (3, 16, 4096, 4)):
        real, n, text = bench.stencil_launches(*args)
        assert (real, n) == (False, 14) and "extract" in text and "scattered" not in text
