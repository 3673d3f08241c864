"""The counting and greedy kernels step through walk elements in 32 bits: no step from below the limit may wrap."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1702_05854_gb300", "csrc")


def test_no_step_wraps():
    header = open(os.path.join(CSRC, "solver.cuh")).read()
    bits = re.search(r"MOST_ENTRIES = \(1ll << (\d+)\) - \(1ll << (\d+)\);", header)
    most = (1 << int(bits[1])) - (1 << int(bits[2]))
    strides = []
    for name in ("cover.cu", "peaks.cu"):
        text = open(os.path.join(CSRC, name)).read()
        for block, cap in re.findall(r"grid_for\((?:[^<;]|\n)*?, (\d+), ([^<;]*?)\), \d+, 0, s>>>", text):
            strides.append(int(block) * eval(cap, {"sm_count": lambda: 152}))
        assert "0xFFFFFFFFll" not in text  # the limit is that one
    assert len(strides) > 30 and most + max(strides) < 1 << 32 and most <= 0xFFFFFFFF
