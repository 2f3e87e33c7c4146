"""Output rows of the step kernel where every CTA has one work item: those of a tile with more than 96 leave 32 at a time, those
of a shorter one row by row, and rows past the end do not."""
import pytest

from paper_2605_16579_b200 import workload
from parity_util import Pair

pytestmark = pytest.mark.gpu


# one and two streams of three heads (a tile that pairs with another head's, and one that does not)
@pytest.mark.parametrize("B,L", [(1, 1), (1, 31), (1, 32), (1, 33), (1, 96), (1, 97), (2, 128), (1, 160), (2, 287), (1, 416)])
def test_rows_at_the_edges_of_a_warp(oracle, B, L):
    cfg = workload.custom(B=B, H=3, D=128, L=L, dtype="bf16", cfg_id=161)
    pair = Pair(oracle, cfg)
    kc, vc, a = workload.commit_inputs(cfg, 0)
    assert pair.commit(kc, vc, a) <= pair.tol
    for step in range(2):
        assert pair.step_full(*workload.step_inputs(cfg, 1, step)) <= pair.tol
