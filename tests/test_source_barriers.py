"""Aligned barrier instructions take a whole warp: every function that issues
one in inline PTX brings its warp together (__syncwarp) first."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2402_11454_gb300", "csrc")


def aligned_barriers():
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.cuh"))):
        text = open(path).read()
        for m in re.finditer(r'asm volatile\("barrier\.[a-z.]*\.aligned', text):
            body = text[text.rfind("\n__device__", 0, m.start()):m.start()]  # the function up to the barrier
            yield os.path.basename(path), text.count("\n", 0, m.start()) + 1, body


def test_aligned_barriers_follow_a_warp_barrier():
    found = list(aligned_barriers())
    assert found  # the cluster path has them
    for name, line, body in found:
        assert "__syncwarp();" in body, f"{name}:{line}"
