"""Calls under stream capture: a graph may be replayed any number of times, or never."""
import pytest
import torch

from paper_2605_16579_b200 import arl2, workload

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _layer(cfg, S, flags=0):
    layer = arl2.Layer(cfg.B, cfg.H, cfg.L, cfg.D, cfg.dtype, device=DEV, flags=flags)
    wq, wk, wv = workload.feature_weights(cfg)
    cos, sin = workload.rope_tables(cfg.L, cfg.D)
    layer.set_params(wq.to(DEV), wk.to(DEV), wv.to(DEV), cos.to(DEV), sin.to(DEV))
    layer.set_state(S)
    return layer


def _cfg(B, H, L, dtype="bf16", D=128):
    cfg = workload.custom(B=B, H=H, D=D, L=L, dtype=dtype, cfg_id=79)
    return cfg, torch.randn(B, H, D, D, generator=torch.Generator().manual_seed(6))


def _capture(fn):
    graph, stream = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph, stream=stream):
        fn()
    torch.cuda.synchronize()
    return graph


def _bits(t):
    return t.clone().view(torch.int16 if t.dtype == torch.bfloat16 else torch.int32)


# more work items than a device has SMs (the second: with its last wave cut into key ranges), and fewer
@pytest.mark.parametrize("B,H,L", [(1, 40, 1560), (1, 40, 1000), (1, 12, 700)])
def test_a_captured_step_is_replayed(B, H, L):
    cfg, S = _cfg(B, H, L)
    layer = _layer(cfg, S)
    q, k, v, g = (t.to(DEV) for t in workload.step_inputs(cfg, 0, 0))
    out = torch.empty(B, L, H, 128, dtype=torch.bfloat16, device=DEV)
    layer.denoise_step(q, k, v, g, out=out)
    torch.cuda.synchronize()
    ref = _bits(out)
    graph = _capture(lambda: layer.denoise_step(q, k, v, g, out=out))
    # (the capture itself has run nothing)
    for _ in range(2):
        out.zero_()
        layer.denoise_step(q, k, v, g, out=out)
        assert torch.equal(_bits(out), ref)
    for _ in range(3):
        out.zero_()
        graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(_bits(out), ref)
    out.zero_()
    layer.denoise_step(q, k, v, g, out=out)
    assert torch.equal(_bits(out), ref)
    layer.sync_status()
