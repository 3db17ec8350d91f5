"""The aligned cluster barriers are undefined where a warp is not together, as after a branch that one thread takes: every one
of them stands directly behind a __syncwarp() or another such barrier, whatever code calls it."""
import glob
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _statements(path):
    text = re.sub(r"/\*.*?\*/|//[^\n]*", "", open(path).read(), flags=re.S)
    return [" ".join(s.split()) for s in re.split(r";(?=\s*\n)|[{}]", text)]


def test_warps_are_together_at_cluster_barriers():
    found = 0
    for path in sorted(glob.glob(os.path.join(ROOT, "paper_2512_23087_b200", "csrc", "*.cu*"))):
        before = ""
        for s in _statements(path):
            if "barrier.cluster" in s:
                found += 1
                assert before == "__syncwarp()" or "barrier.cluster" in before, f"{os.path.basename(path)}: {s}"
            before = s
    assert found >= 4
