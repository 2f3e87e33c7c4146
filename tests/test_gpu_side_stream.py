"""Token-level pass: the stream beside the caller's keeps out of other captures."""
import pytest
import torch

from graph_util import graph_roots
from paper_2605_16579_b200 import arl2, workload

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
CFG = workload.custom(B=1, H=4, D=128, L=700, dtype="bf16", cfg_id=77)   # a shape that forks


def _layer():
    layer = arl2.Layer(CFG.B, CFG.H, CFG.L, CFG.D, CFG.dtype, device=DEV)
    wq, wk, wv = workload.feature_weights(CFG)
    cos, sin = workload.rope_tables(CFG.L, CFG.D)
    layer.set_params(wq.to(DEV), wk.to(DEV), wv.to(DEV), cos.to(DEV), sin.to(DEV))
    layer.set_state(torch.randn(CFG.B, CFG.H, 128, 128, generator=torch.Generator().manual_seed(3)))
    return layer


def _inputs(seed):
    q, k, v, g = (t.to(DEV) for t in workload.step_inputs(CFG, seed, 0))
    return q, k, v, g, workload.token_gate_logits(CFG, seed)[0].to(DEV)


def _out():
    return torch.zeros(CFG.B, CFG.L, CFG.H, CFG.D, dtype=torch.bfloat16, device=DEV)


def _same(a, b):
    return torch.equal(a.view(torch.int16), b.view(torch.int16))


def test_a_context_destroyed_in_an_open_capture_and_the_next_one():
    x = _inputs(0)
    first, second = _layer(), _layer()
    ref, captured, eager = _out(), _out(), _out()
    first.denoise_step_token_level(*x, out=ref)        # takes its second stream here
    buffers = (first.state, first.workspace)           # (the graph goes on using them)
    torch.cuda.synchronize()
    s_cap, s_run = torch.cuda.Stream(), torch.cuda.Stream()
    graph = torch.cuda.CUDAGraph(keep_graph=True)
    with torch.cuda.graph(graph, stream=s_cap):
        first.denoise_step_token_level(*x, out=captured)
        first.close()
        with torch.cuda.stream(s_run):
            second.denoise_step_token_level(*x, out=eager)
    assert graph_roots(graph) == 2
    graph.replay()
    torch.cuda.synchronize()
    assert _same(captured, ref) and _same(eager, ref)
    second.sync_status()
    third = _layer()                                   # the capture is over: its stream may be handed out again
    again = _out()
    third.denoise_step_token_level(*x, out=again)
    third.sync_status()
    assert _same(again, ref)
    del buffers


def test_a_call_beside_an_open_capture_of_the_same_context():
    x = _inputs(1)
    layer = _layer()
    ref, captured, eager = _out(), _out(), _out()
    layer.denoise_step_token_level(*x, out=ref)
    torch.cuda.synchronize()
    s_cap, s_run = torch.cuda.Stream(), torch.cuda.Stream()
    graph = torch.cuda.CUDAGraph(keep_graph=True)
    with torch.cuda.graph(graph, stream=s_cap):
        layer.denoise_step_token_level(*x, out=captured)
        with torch.cuda.stream(s_run):
            layer.denoise_step_token_level(*x, out=eager)
        layer.denoise_step_token_level(*x, out=captured)
    torch.cuda.synchronize()
    graph.replay()
    torch.cuda.synchronize()
    assert _same(captured, ref) and _same(eager, ref)
    layer.sync_status()
