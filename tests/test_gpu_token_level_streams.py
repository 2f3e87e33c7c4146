"""Token-level pass: the route with a stream of the context's own beside the caller's gives the bits of the route without."""
import pytest
import torch

from paper_2605_16579_b200 import arl2, workload

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _layer(cfg, S):
    layer = arl2.Layer(cfg.B, cfg.H, cfg.L, cfg.D, cfg.dtype, device=DEV)
    wq, wk, wv = workload.feature_weights(cfg)
    cos, sin = workload.rope_tables(cfg.L, cfg.D)
    layer.set_params(wq.to(DEV), wk.to(DEV), wv.to(DEV), cos.to(DEV), sin.to(DEV))
    layer.set_state(S)
    return layer


@pytest.mark.parametrize("B,H,L", [(1, 4, 700), (2, 3, 900), (1, 12, 1560), (1, 2, 640), (1, 40, 1560)])
def test_forked_and_single_stream_routes_agree(B, H, L):
    # forked: runs of tiles (more than 5 to a head) and a softmax branch on at most 111 of 148 SMs; the fourth shape goes
    # by whole heads and the last one fills the device: no fork, whatever the call
    cfg = workload.custom(B=B, H=H, D=128, L=L, dtype="bf16", cfg_id=76)
    S = torch.randn(B, H, 128, 128, generator=torch.Generator().manual_seed(3))
    q, k, v, g = (t.to(DEV) for t in workload.step_inputs(cfg, 0, 0))
    alpha = workload.token_gate_logits(cfg, 0)[0].to(DEV)
    # a first call under capture finds no side stream and stays on the caller's
    single = _layer(cfg, S)
    out = torch.empty(B, L, H, 128, dtype=torch.bfloat16, device=DEV)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    stream = torch.cuda.Stream()
    with torch.cuda.graph(graph, stream=stream):
        single.denoise_step_token_level(q, k, v, g, alpha, out=out)
    graph.replay()
    torch.cuda.synchronize()
    ref = out.clone()
    # eager calls on two streams by two contexts, twice each, and a capture once the side stream is there
    forked = [_layer(cfg, S), _layer(cfg, S)]
    outs = [torch.empty_like(out) for _ in range(4)]
    torch.cuda.synchronize()
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    for i in range(4):
        with torch.cuda.stream(streams[i & 1]):
            forked[i & 1].denoise_step_token_level(q, k, v, g, alpha, out=outs[i])
    torch.cuda.synchronize()
    graph2 = torch.cuda.CUDAGraph()
    out.zero_()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph2, stream=stream):
        forked[0].denoise_step_token_level(q, k, v, g, alpha, out=out)
    graph2.replay()
    torch.cuda.synchronize()
    for o in outs + [out]:
        assert torch.equal(o.view(torch.int16), ref.view(torch.int16))
    for layer in [single] + forked:
        layer.sync_status()
