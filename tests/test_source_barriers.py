"""Barriers that the kernels' sources must hold, whatever a compiler makes of
them today.  Aligned barrier instructions take a whole warp: every function
that issues one in inline PTX brings its warp together (__syncwarp) first.  A
table that several lanes clear is used by them only after a barrier: votes and
shuffles do not order shared memory."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2402_11454_gb300", "csrc")


def sources():
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.cuh"))):
        yield path, open(path).read()


def aligned_barriers():
    for path, text in sources():
        for m in re.finditer(r'asm volatile\("barrier\.[a-z.]*\.aligned', text):
            body = text[text.rfind("\n__device__", 0, m.start()):m.start()]  # the function up to the barrier
            yield os.path.basename(path), text.count("\n", 0, m.start()) + 1, body


def test_aligned_barriers_follow_a_warp_barrier():
    found = list(aligned_barriers())
    assert found  # the cluster path has them
    for name, line, body in found:
        assert "__syncwarp();" in body, f"{name}:{line}"


def test_tables_cleared_by_many_lanes_are_used_after_a_barrier():
    found = 0
    for path, text in sources():
        for m in re.finditer(r"for \([^\n]*\) (\w*tab)\.clear\(\w+\);", text):
            found += 1
            use = re.compile(r"\b%s\b" % m.group(1)).search(text, m.end())
            end = use.start() if use else len(text)
            assert re.search(r"__sync(warp|threads)\(", text[m.end():end]), \
                "%s:%d" % (os.path.basename(path), text.count("\n", 0, m.start()) + 1)
    assert found >= 4
