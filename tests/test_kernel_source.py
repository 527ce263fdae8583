"""Properties of the kernel sources that no run can show."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2507_01770_gb300", "csrc")


def _code(path):
    return re.sub(r"//[^\n]*", "", open(path).read())


def test_a_word_that_other_warps_write_is_read_once_for_the_warp():
    # Lanes that each read such a word may see different values; a branch on
    # it around a full-mask ballot or shuffle would then leave lanes behind.
    # One lane's read reaches the others through a warp-wide exchange in the
    # statement that reads it.
    reads = 0
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        for stmt in re.split(r"[;{}]", _code(path)):
            if re.search(r"\*\s*\(\s*(const\s+)?volatile\b", stmt):
                reads += 1
                assert re.search(r"__(shfl|any|all|ballot)_sync\s*\(", stmt) and "lane == 0" in stmt, (path, stmt.strip())
    assert reads
