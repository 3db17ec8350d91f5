"""Aligned instructions are undefined where a warp is not together, as after a branch that some of its threads take: every
cluster barrier and every read of tensor memory stands directly behind a __syncwarp() or another such instruction, whatever
code calls it."""
import glob
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _statements(path):
    text = re.sub(r"/\*.*?\*/|//[^\n]*", "", open(path).read(), flags=re.S)
    return [" ".join(s.split()) for s in re.split(r";(?=\s*\n)|[{}]", text)]


ALIGNED = ("barrier.cluster", "tcgen05.ld.sync", "tcgen05.wait::ld.sync")


def _aligned(statement):
    return any(name in statement for name in ALIGNED)


def test_warps_are_together_at_aligned_instructions():
    found = 0
    for path in sorted(glob.glob(os.path.join(ROOT, "paper_2512_23087_b200", "csrc", "*.cu*"))):
        before = ""
        for s in _statements(path):
            if _aligned(s):
                found += 1
                assert before == "__syncwarp()" or _aligned(before), f"{os.path.basename(path)}: {s}"
            before = s
    assert found >= 6
