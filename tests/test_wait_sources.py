"""What the sources say of waits that expire: a warp's lanes stay together, and nothing is left in flight.

The lanes of a warp vote, shuffle and synchronise further down; one that had given up by itself would be missing there, and
the others would wait for it without a limit.  An expiry that splits a warp cannot be brought about at will, and must not be
on a GPU, so the sources are looked at.
"""
import glob
import os
import re

from test_overlapped_launch_sources import CSRC, _code, _kernels

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


# In these the flag is looked at behind a barrier that every thread passes after its last wait.
_BEHIND_A_BARRIER = {"tc_token_prepare_kernel", "tc_token_readout_kernel", "tc_gemm_pair_kernel"}


def _on_the_flag(body):
    """Whether a wait for copies or MMAs in flight depends on the flag that another role may yet raise."""
    for m in re.finditer(r"if \([^{};]*abort_flag[^{};]*\)\s*\{", body):
        depth, i = 1, m.end()
        while depth:
            depth += {"{": 1, "}": -1}.get(body[i], 0)
            i += 1
        if "drain_bar(" in body[m.end():i]:
            return True
    return False


def test_what_is_in_flight_is_waited_for_in_any_case():
    """A role that is through does not know whether another one will give up on what it sent for."""
    seen = 0
    for path in sorted(glob.glob(os.path.join(CSRC, "arl2_tc*.cu"))):
        for name, _, body in _kernels(_code(path)):
            if "drain_bar(" in body and name not in _BEHIND_A_BARRIER:
                seen += 1
                assert not _on_the_flag(body), (os.path.basename(path), name)
    assert seen >= 4


def test_a_wait_that_depends_on_the_flag_is_noticed():
    assert _on_the_flag("if (!ok || __any_sync(0xffffffffu, *abort_flag)) { commit(b); drain_bar(b, 0); }")
    assert not _on_the_flag("if (!ok || *abort_flag) { stop(); } drain_bar(b, 0);")
