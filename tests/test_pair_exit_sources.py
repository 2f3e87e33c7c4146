"""What a kernel on pairs of CTAs waits for before it ends.

A commit of the MMAs arrives on a barrier of both CTAs.  That the first CTA has seen its own arrival does not order the
other's, so a CTA that ends without a wait of its own may be gone when the arrival reaches its shared memory.  No run shows
that reliably, so the source is looked at.
"""
import os
import re

from test_overlapped_launch_sources import CSRC, _code, _kernels


def _outside_rank_blocks(body):
    """The body without the statements and blocks that only one CTA of a pair runs (`if (rank ...)`)."""
    out, i = "", 0
    for m in re.finditer(r"if \(rank\b", body):
        if m.start() < i:
            continue
        out += body[i:m.start()]
        depth, j = 1, body.index("(", m.start()) + 1
        while depth:
            depth += {"(": 1, ")": -1}.get(body[j], 0)
            j += 1
        j += len(body[j:]) - len(body[j:].lstrip())
        if body[j] == "{":
            depth, j = 1, j + 1
            while depth:
                depth += {"{": 1, "}": -1}.get(body[j], 0)
                j += 1
        else:
            j = body.index(";", j) + 1
        i = j
    return out + body[i:]


def _unwaited(body):
    """Barriers that a commit to both CTAs arrives on and that not every CTA waits for."""
    committed = set(re.findall(r"mma_commit_pair_if\([^;]*?(k\w*Bar[A-Za-z]+)", body))
    waited = set(re.findall(r"(?:wait_bar|wait_bar_warp|drain_bar)\([^;]*?(k\w*Bar[A-Za-z]+)", _outside_rank_blocks(body)))
    return committed, committed - waited


def test_both_ctas_of_a_pair_wait_for_every_barrier_they_share():
    seen = 0
    for name in sorted(os.listdir(CSRC)):
        if name.endswith(".cu"):
            for kernel, _, body in _kernels(_code(os.path.join(CSRC, name))):
                committed, missing = _unwaited(body)
                seen += len(committed)
                assert not missing, (name, kernel, missing)
    assert seen >= 3


def test_the_stages_last_given_back_are_waited_for():
    """The producers' loop waits for a stage only when it is wanted again: the last ones need a loop of their own behind it."""
    body = dict((k, b) for k, _, b in _kernels(_code(os.path.join(CSRC, "arl2_tc_gemm.cu"))))["tc_gemm_pair_kernel"]
    producer = _outside_rank_blocks(body[:body.index("*asked = n;")])
    waits = [m.start() for m in re.finditer(r"wait_bar\(bars \+ 8 \* \(kGPBarEmpty0", producer)]
    assert len(waits) == 2 and waits[1] > producer.rindex("tma_load_2d_pair")


def test_a_wait_of_one_cta_only_is_noticed():
    body = "if (rank == 0) { mma_commit_pair_if(lead, bars + 8 * kXBarEnd); drain_bar(bars + 8 * kXBarEnd, 0); } cluster_sync_all();"
    assert _unwaited(body)[1] == {"kXBarEnd"}
    assert _unwaited(body.replace("drain_bar(bars + 8 * kXBarEnd, 0); }", "} drain_bar(bars + 8 * kXBarEnd, 0);"))[1] == set()
