"""Token-level pass: its second stream has the priority of the caller's."""
import pytest
import torch

from graph_util import graph_roots, kernel_priorities
from test_gpu_side_stream import _inputs, _layer, _out, _same

pytestmark = pytest.mark.gpu


def test_the_second_stream_has_the_priority_of_the_callers():
    x = _inputs(2)
    layer = _layer()
    ref = _out()
    layer.denoise_step_token_level(*x, out=ref)        # on the default stream
    torch.cuda.synchronize()
    high, low = torch.cuda.Stream(priority=-1), torch.cuda.Stream()
    assert high.priority < low.priority
    for stream in (high, low, high):
        out, eager = _out(), _out()
        torch.cuda.synchronize()
        with torch.cuda.stream(stream):
            layer.denoise_step_token_level(*x, out=eager)
        graph = torch.cuda.CUDAGraph(keep_graph=True)
        with torch.cuda.graph(graph, stream=stream):
            layer.denoise_step_token_level(*x, out=out)
        assert graph_roots(graph) == 2
        assert set(kernel_priorities(graph)) == {stream.priority}
        graph.replay()
        torch.cuda.synchronize()
        assert _same(out, ref) and _same(eager, ref)
    # straight into a capture on a stream of another priority
    graph = torch.cuda.CUDAGraph(keep_graph=True)
    with torch.cuda.graph(graph, stream=low):
        layer.denoise_step_token_level(*x, out=out)
    assert graph_roots(graph) == 2
    assert set(kernel_priorities(graph)) == {low.priority}
    layer.sync_status()
