"""A wait that expires ends a warp's role for all lanes alike.

The lanes of a warp vote, shuffle and synchronise further down; one that had given up by itself would be missing there, and
the others would wait for it without a limit.  An expiry that splits a warp cannot be brought about at will, and must not be
on a GPU, so the sources are looked at.
"""
import glob
import os
import re

from test_overlapped_launch_sources import CSRC, _code

# a lane's own wait whose end by time-out leaves the function
_LEAVES = re.compile(r"!\s*wait_bar\((?:[^()]|\([^()]*\)|\((?:[^()]|\([^()]*\))*\))*\)\s*\)\s*(?:\{\s*)?return")


def test_no_lane_leaves_by_itself():
    looked_at, bad = 0, []
    for path in sorted(glob.glob(os.path.join(CSRC, "arl2_tc*.cu"))):
        code = _code(path)
        looked_at += code.count("wait_bar_warp(")
        bad += [f"{os.path.basename(path)}: {m.group(0)}" for m in _LEAVES.finditer(code)]
    assert looked_at >= 10
    assert not bad, bad


def test_a_lane_that_leaves_is_noticed():
    for text in ("if (!wait_bar(bar_s, n & 1, ab, 20 + t)) return;", "if (i > 0 && !wait_bar(bars + 8 * (kBarO0 + t), 0, ab, 1)) {\n  return;"):
        assert _LEAVES.search(text)
        assert not _LEAVES.search(text.replace("wait_bar(", "wait_bar_warp("))
    assert not _LEAVES.search("if (!wait_bar(bar, 0, ab, 1)) ok = false;")
