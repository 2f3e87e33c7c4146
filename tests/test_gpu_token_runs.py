"""commit_tokens where few heads leave SMs idle: the chunks of a head walked in runs side by side, which are put together
at the end (S -> M S + N per run).  Sizes on either side of the rule's lines: two runs with a slab of columns per SM and
with two, three runs, four, a shorter last run that ends inside a chunk."""
import numpy as np
import pytest
import torch

from paper_2605_16579_b200 import arl2, workload
from parity_util import Pair

pytestmark = pytest.mark.gpu
FLAG = arl2.ARL2_FLAG_TOKEN_GATES


@pytest.mark.parametrize("B,H,L,decayed", [
    (1, 2, 2100, False),     # two runs of 17 and 16 chunks, the last of 52 tokens
    (2, 3, 2000, True),      # two runs, the most heads whose slabs have an SM each
    (1, 7, 3000, False),     # two runs, two slabs to an SM
    (1, 2, 4680, False),     # three runs
    (1, 1, 8000, True),      # four runs
])
def test_runs_match_the_token_loop(oracle, B, H, L, decayed):
    cfg = workload.custom(B=B, H=H, D=128, L=L, dtype="bf16", cfg_id=141)
    pair = Pair(oracle, cfg, flags=FLAG | (arl2.ARL2_FLAG_DELTA_DECAYED_PREDICTION if decayed else 0))
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
