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


@pytest.mark.parametrize("kind", ["commit", "delta", "decay", "tokens", "clean"])
def test_a_captured_block_is_replayed(kind):
    """Two denoise passes and the state update: every replay reads the state that the one before left."""
    cfg, S = _cfg(2, 3, 300)
    flags = arl2.ARL2_FLAG_TOKEN_GATES if kind == "tokens" else 0
    q, k, v, g = (t.to(DEV) for t in workload.step_inputs(cfg, 0, 0))
    kc, vc, a = (t.to(DEV) for t in workload.commit_inputs(cfg, 0))
    alpha, beta = (t.to(DEV) for t in workload.token_gate_logits(cfg, 0))
    eager, captured = _layer(cfg, S, flags), _layer(cfg, S, flags)

    def block(layer, outs):
        layer.denoise_step(q, k, v, g, out=outs[0])
        layer.denoise_step(k, q, v, g, out=outs[1])
        if kind == "commit":
            layer.commit(kc, vc, a)
        elif kind == "delta":
            layer.commit_delta(kc, vc, a, beta)
        elif kind == "decay":
            layer.commit_decay_tokens(kc, vc, alpha)
        elif kind == "tokens":
            layer.commit_tokens(kc, vc, alpha, beta)
        else:
            layer.clean_pass(q, kc, vc, g, a, out=outs[2])

    outs_e, outs_c = ([torch.zeros_like(q) for _ in range(3)] for _ in range(2))
    graph = _capture(lambda: block(captured, outs_c))   # (has run nothing: the state is as it was)
    for i in range(5):
        block(eager, outs_e)
        if i in (0, 4):                                  # eager calls before and after the replays
            block(captured, outs_c)
        else:
            graph.replay()
        torch.cuda.synchronize()
        for e, c in zip(outs_e, outs_c):
            assert torch.equal(_bits(e), _bits(c)), f"block {i}"
        assert torch.equal(_bits(eager.state), _bits(captured.state)), f"block {i}"
    for layer in (eager, captured):
        layer.sync_status()
