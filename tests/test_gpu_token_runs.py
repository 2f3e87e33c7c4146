"""commit_tokens where few heads leave SMs idle: the chunks of a head walked in runs side by side, which are put together
at the end (S -> M S + N per run).  Sizes on either side of the rule's lines: two runs with a slab of columns per SM and
with two, three runs, four, a shorter last run that ends inside a chunk."""
import numpy as np
import pytest
import torch

from graph_util import captured_kernels
from paper_2605_16579_b200 import arl2, workload
from parity_util import Pair

pytestmark = pytest.mark.gpu
FLAG = arl2.ARL2_FLAG_TOKEN_GATES


def _runs(layer, cfg, inputs):
    """(runs, slabs of 16 columns per CTA) of the walk that the call launches (1 run without a join)."""
    seen = [k for k in captured_kernels(lambda: layer.commit_tokens(*inputs)) if "tc_token_scan_kernel" in k[0] or "tc_token_join_kernel" in k[0]]
    name, grid, block, _ = seen[0]
    slabs = (block[0] - 32) // 128
    runs = (grid[0] * slabs // 8 + 1) // 2
    assert len(seen) == (2 if runs > 1 else 1) and grid[1:] == (cfg.H, cfg.B)
    return runs, slabs


@pytest.mark.parametrize("B,H,L,decayed,runs,slabs", [
    (1, 2, 2100, False, 2, 1),     # runs of 17 and 16 chunks, the last of 52 tokens
    (2, 3, 2000, True, 2, 1),      # the most heads of which two runs have an SM per slab
    (1, 12, 2300, False, 2, 2),    # two slabs to a CTA
    (1, 7, 3000, False, 3, 2),
    (1, 2, 4680, False, 3, 1),
    (1, 1, 8000, True, 4, 1),
    (1, 12, 1560, False, 1, 1),    # beside the rule's lines: too few chunks, and no SM left
    (1, 13, 3000, True, 1, 1),
])
def test_runs_match_the_token_loop(oracle, B, H, L, decayed, runs, slabs):
    cfg = workload.custom(B=B, H=H, D=128, L=L, dtype="bf16", cfg_id=141)
    pair = Pair(oracle, cfg, flags=FLAG | (arl2.ARL2_FLAG_DELTA_DECAYED_PREDICTION if decayed else 0))
    kc, vc, _ = workload.commit_inputs(cfg, 7)
    on = [t.to(pair.dev) for t in (kc, vc, *workload.token_gate_logits(cfg, 7))]
    saved = pair.layer.get_state()
    assert _runs(pair.layer, cfg, on) == (runs, slabs)
    pair.layer.set_state(saved)
    for blk, (am, bm) in enumerate([(7.0, 0.0), (9.0, 2.0), (2.0, 0.0)]):   # ordinary, hardly any, strong forgetting
        kc, vc, _ = workload.commit_inputs(cfg, blk)
        alpha, beta = workload.token_gate_logits(cfg, blk, alpha_mean=am, beta_mean=bm)
        err = pair.commit_tokens(kc, vc, alpha, beta, decayed_prediction=decayed)
        assert err <= pair.tol, f"block {blk}: error {err:.3e} > {pair.tol}"
    q, k, v, g = workload.step_inputs(cfg, 3, 0)
    assert pair.step_full(q, k, v, g) <= pair.tol      # the operand copy of S was written too


def test_runs_with_keys_of_a_common_direction(oracle):
    """What a run carries over is nearly singular then, and the entering state is almost wholly replaced."""
    cfg = workload.custom(B=1, H=3, D=128, L=2200, dtype="bf16", cfg_id=142)
    pair = Pair(oracle, cfg, flags=FLAG)
    gen = torch.Generator().manual_seed(5)
    for blk in range(2):
        kc, vc, _ = workload.commit_inputs(cfg, blk)
        kc = (0.3 * kc.float() + torch.randn(1, 1, 3, 128, generator=gen)).to(torch.bfloat16)
        alpha, beta = workload.token_gate_logits(cfg, blk, alpha_mean=8.0, beta_mean=1.0)
        assert pair.commit_tokens(kc, vc, alpha, beta) <= pair.tol


def test_an_expired_wait_in_the_last_run_leaves_the_state(oracle):
    cfg = workload.custom(B=1, H=2, D=128, L=2100, dtype="bf16", cfg_id=143)
    pair = Pair(oracle, cfg, flags=FLAG)
    kc, vc, _ = workload.commit_inputs(cfg, 0)
    alpha, beta = workload.token_gate_logits(cfg, 0)
    assert pair.commit_tokens(kc, vc, alpha, beta) <= pair.tol
    saved = pair.layer.get_state()
    on = [t.to(pair.dev) for t in (kc, vc, alpha, beta)]
    pair.layer.debug_set_walk_wait_limit(0)
    pair.layer.commit_tokens(*on)
    with pytest.raises(arl2.Arl2Error):
        pair.layer.sync_status()
    assert torch.equal(pair.layer.get_state(), saved)
    pair.layer.debug_set_walk_wait_limit(-1)
    kc, vc, _ = workload.commit_inputs(cfg, 1)
    alpha, beta = workload.token_gate_logits(cfg, 1)
    assert pair.commit_tokens(kc, vc, alpha, beta) <= pair.tol
    pair.layer.sync_status()
