"""The plain-FMA step on clusters of CTAs that share a 16-row unit: edges of key tiles, CTAs without keys, both splits."""
import pytest
import torch

from paper_2605_16579_b200 import arl2, workload
from parity_util import Pair, TOL, head_errors

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype,D,B,H,L", [
    # four CTAs per unit (units of 16 rows x 4 within 7/8 of 148 SMs): key tiles of 64
    ("fp32", 64, 1, 1, 65), ("fp32", 64, 1, 2, 128), ("fp32", 64, 1, 2, 193), ("fp32", 64, 1, 1, 512),
    ("fp32", 128, 1, 1, 65), ("fp32", 128, 2, 1, 255), ("bf16", 64, 1, 2, 250),
    # two CTAs per unit: key tiles of 128
    ("fp32", 64, 1, 4, 129), ("fp32", 64, 3, 1, 321), ("fp32", 128, 1, 2, 400), ("bf16", 64, 2, 2, 250),
    # one: the smallest sequences, and just past the two-CTA line
    ("fp32", 64, 1, 1, 64), ("fp32", 64, 1, 5, 208),
])
def test_step_on_clusters(oracle, dtype, D, B, H, L):
    cfg = workload.custom(B=B, H=H, D=D, L=L, dtype=dtype, cfg_id=74)
    pair = Pair(oracle, cfg)
    kc, vc, a = workload.commit_inputs(cfg, 0)
    assert pair.commit(kc, vc, a) <= pair.tol
    q, k, v, g = workload.step_inputs(cfg, 1, 0)
    assert pair.step_full(q, k, v, g) <= pair.tol
    assert pair.step_full(q, k, v, torch.full_like(g, -40.0)) <= pair.tol


@pytest.mark.parametrize("D,H,L", [(64, 2, 100), (64, 3, 300), (128, 2, 100)])
def test_step_on_clusters_without_maps(oracle, D, H, L):
    cfg = workload.custom(B=1, H=H, D=D, L=L, dtype="fp32", cfg_id=75)
    layer = arl2.Layer(1, H, L, D, "fp32", device="cuda:0")
    S = torch.randn(1, H, D, D, generator=torch.Generator().manual_seed(5))
    layer.set_state(S)
    q, k, v, g = workload.step_inputs(cfg, 0, 0)
    got = layer.denoise_step(q.cuda(), k.cuda(), v.cuda(), g.cuda()).cpu().numpy()
    layer.sync_status()
    eye = torch.eye(D).expand(H, D, D).contiguous()
    ref = oracle.step(q, k, v, g, S.double().numpy(), eye, torch.ones(L, D // 2), torch.zeros(L, D // 2))
    assert float(head_errors(got, ref).max()) <= TOL["fp32"]
