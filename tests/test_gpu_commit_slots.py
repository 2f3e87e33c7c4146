"""Commits whose heads fall into so many runs of tiles that the finishing kernel takes the slots in several batches (6 slots
for the gated-linear rule, 4 and a second set beside the first for the delta rule)."""
import pytest

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
