"""Commits whose heads fall into so many runs of tiles that the finishing kernel takes the slots in several batches (6 slots
for the gated-linear rule, 4 and a second set beside the first for the delta rule)."""
import pytest

from graph_util import captured_kernels
from paper_2605_16579_b200 import workload
from parity_util import Pair

pytestmark = pytest.mark.gpu


# three heads of 1, 7, 8, 9, 12, 13, 17 and 26 tiles in runs of two, which cross from head to head: 1 to 14 slots per head
@pytest.mark.parametrize("L", [100, 800, 1024, 1100, 1536, 1600, 2100, 3300])
def test_slots_in_batches(oracle, L):
    cfg = workload.custom(B=1, H=3, D=128, L=L, dtype="bf16", cfg_id=151)
    pair = Pair(oracle, cfg)
    for blk in range(2):
        kc, vc, a = workload.commit_inputs(cfg, blk)
        assert pair.commit(kc, vc, a) <= pair.tol
        kc, vc, a = workload.commit_inputs(cfg, blk + 10)
        assert pair.commit_delta(kc, vc, a, workload.beta_logits(cfg, blk)) <= pair.tol
    q, k, v, g = workload.step_inputs(cfg, 2, 0)
    assert pair.step_full(q, k, v, g) <= pair.tol


# The finishing kernel with room for four CTAs per SM: more than three to an SM, or with per-token decay more than one (148
# SMs, 8 CTAs per head).  Slots per head: 1 and 2; with decay 7 (one after the first six), 4, 1 and 2.
@pytest.mark.parametrize("rule,B,H,L,many", [
    ("commit", 7, 8, 100, True), ("commit", 3, 24, 218, True), ("commit", 8, 8, 300, True), ("commit", 5, 11, 130, False),
    ("decay", 1, 20, 2100, True), ("decay", 1, 19, 1000, True), ("decay", 4, 8, 100, True), ("decay", 3, 6, 300, False),
])
def test_many_heads(oracle, rule, B, H, L, many):
    cfg = workload.custom(B=B, H=H, D=128, L=L, dtype="bf16", cfg_id=152)
    pair = Pair(oracle, cfg)
    heads = [(0, 0), (0, H - 1), (B // 2, H // 2), (B - 1, 0), (B - 1, H - 1)]
    for blk in range(2):
        kc, vc, a = workload.commit_inputs(cfg, blk)
        alpha = workload.token_gate_logits(cfg, blk)[0]
        err = pair.commit_decay_tokens(kc, vc, alpha, heads=heads) if rule == "decay" else pair.commit(kc, vc, a, heads=heads)
        assert err <= pair.tol
    on = [t.to(pair.dev) for t in (kc, vc, alpha if rule == "decay" else a)]
    call = pair.layer.commit_decay_tokens if rule == "decay" else pair.layer.commit
    names = [k[0] for k in captured_kernels(lambda: call(*on)) if "tc_commit_finish_kernel" in k[0]]
    assert len(names) == 1 and ("ILi0ELb1EE" if many else "ILi0ELb0EE") in names[0]
