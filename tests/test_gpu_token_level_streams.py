"""Token-level pass: the route with a stream of the context's own beside the caller's gives the bits of the route without."""
import pytest
import torch

from graph_util import graph_roots
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


@pytest.mark.parametrize("B,H,L,forks", [(1, 4, 700, True), (2, 3, 900, True), (1, 12, 1560, True), (1, 2, 640, False), (1, 40, 1560, False)])
def test_route_and_order_of_the_passes(B, H, L, forks):
    """Which shapes fork, and that a pass waits for what its stream does before it: the inputs of every pass arrive on the
    caller's stream behind a kernel of a millisecond, in the buffers of the pass before, and a commit moves the state on
    between the passes, so that a branch that starts early or is not waited for gives other bits."""
    cfg = workload.custom(B=B, H=H, D=128, L=L, dtype="bf16", cfg_id=78)
    S = torch.randn(B, H, 128, 128, generator=torch.Generator().manual_seed(4))
    steps = []
    for i in range(4):
        q, k, v, g = workload.step_inputs(cfg, i, 0)
        steps.append([t.to(DEV) for t in (q, k, v, g, workload.token_gate_logits(cfg, i)[0], workload.commit_inputs(cfg, i)[2])])
    bufs = [torch.empty_like(t) for t in steps[0]]
    out = torch.empty(B, L, H, 128, dtype=torch.bfloat16, device=DEV)

    def one(layer):
        layer.denoise_step_token_level(*bufs[:5], out=out)
        layer.commit(bufs[1], bufs[2], bufs[5])

    def fill(i):
        for b, t in zip(bufs, steps[i]):
            b.copy_(t)

    # the reference: a first call under capture, which stays on one stream, replayed with a synchronisation around each pass
    single = _layer(cfg, S)
    fill(0)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph(keep_graph=True)
    stream = torch.cuda.Stream()
    with torch.cuda.graph(graph, stream=stream):
        single.denoise_step_token_level(*bufs[:5], out=out)
    assert graph_roots(graph) == 1
    refs = []
    for i in range(4):
        fill(i)
        torch.cuda.synchronize()
        graph.replay()
        torch.cuda.synchronize()
        refs.append(out.clone())
        single.commit(bufs[1], bufs[2], bufs[5])
        torch.cuda.synchronize()
    ref_state = single.get_state()
    # eager passes, nothing waited for by the host
    layer = _layer(cfg, S)
    outs = [torch.empty_like(out) for _ in range(4)]
    torch.cuda.synchronize()
    with torch.cuda.stream(stream):
        for i in range(4):
            torch.cuda._sleep(2_000_000)
            fill(i)
            one(layer)
            outs[i].copy_(out)
    torch.cuda.synchronize()
    for o, r in zip(outs, refs):
        assert torch.equal(o.view(torch.int16), r.view(torch.int16))
    assert torch.equal(layer.get_state(), ref_state)
    # and which way such a context goes
    graph = torch.cuda.CUDAGraph(keep_graph=True)
    with torch.cuda.graph(graph, stream=stream):
        layer.denoise_step_token_level(*bufs[:5], out=out)
    assert graph_roots(graph) == (2 if forks else 1)
    for x in (single, layer):
        x.sync_status()
