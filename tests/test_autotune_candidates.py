"""The autotuner's launch shapes are ones the stacking kernel runs as they are: a
block holds at most KMAX_THREADS / 32 warps, and a candidate of more would time one
of the others again and could be returned in its place.  Checked in the source (no GPU)."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2609_01897_gb300", "csrc")


def test_candidates_fit_the_kernel():
    stack = open(os.path.join(CSRC, "vista_stack.cuh")).read()
    tune = open(os.path.join(CSRC, "vista_autotune.cu")).read()
    most = int(re.search(r"KMAX_THREADS = (\d+);", stack).group(1)) // 32
    warps = [int(x) for x in re.findall(r"\badd\(\w+, \w+, (\d+), \w+\)", tune)]
    assert len(warps) >= 2 and max(warps) <= most, (warps, most)
