"""Output rows of the token-level readout: they come and leave 32 at a time, and rows past the end do neither."""
import numpy as np
import pytest

from paper_2605_16579_b200 import workload
from parity_util import Pair, head_errors

pytestmark = pytest.mark.gpu


# up to one tile, and several tiles per CTA (the next tile's state goes where these rows leave from)
@pytest.mark.parametrize("B,L", [(1, 1), (1, 31), (1, 32), (1, 33), (2, 96), (1, 97), (2, 128), (1, 129), (2, 287), (1, 416)])
def test_rows_at_the_edges_of_a_warp(oracle, B, L):
    cfg = workload.custom(B=B, H=3, D=128, L=L, dtype="bf16", cfg_id=181)
    pair = Pair(oracle, cfg)
    kc, vc, a = workload.commit_inputs(cfg, 0)
    assert pair.commit(kc, vc, a) <= pair.tol
    d = pair.dev
    for step in range(2):
        q, k, v, g = workload.step_inputs(cfg, 1, step)
        alpha = workload.token_gate_logits(cfg, 1)[0]
        pair.g_out.t.fill_(float("nan"))
        out = pair.layer.denoise_step_token_level(q.to(d), k.to(d), v.to(d), g.to(d), alpha.to(d), out=pair.g_out.t)
        got = out.float().cpu().numpy()
        pair.check_guards()
        ref = oracle.step_token_level(q, k, v, g, pair.S_ref, alpha, pair.wq, pair.wk, pair.wv, pair.cos, pair.sin)
        assert np.isfinite(got).all()
        assert float(head_errors(got, ref).max()) <= pair.tol
    pair.layer.sync_status()
