"""Warp collectives name their lanes in a mask, so every named lane must reach
them: none may stand on the right of a short-circuit, where lanes that disagree
about the left side would leave the others waiting."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1912_03998_gb300", "csrc")
BEHIND = re.compile(r"(?:\|\||&&)[^;{}]*?__(?:shfl\w*|ballot|any|all|match_\w+|reduce_\w+)_sync")


def code(path):
    s = open(path).read()
    s = re.sub(r"//[^\n]*", "", s)
    return re.sub(r"/\*.*?\*/", "", s, flags=re.S)


def test_no_collective_behind_a_short_circuit():
    assert BEHIND.search("if (sp > n || __shfl_sync(m, b -= k, l) < 0) return;")
    files = sorted(glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.cuh")))
    assert files
    for f in files:
        hits = [m.group(0) for m in BEHIND.finditer(code(f))]
        assert not hits, f"{os.path.basename(f)}: {hits}"
