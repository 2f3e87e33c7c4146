"""A launch that is refused is reported by its own call and by no other."""
import pytest
import torch

from paper_2605_16579_b200 import arl2, workload

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("dtype,D", [("bf16", 128), ("fp32", 64)])
def test_a_refused_launch_does_not_fail_the_next_call(dtype, D):
    cfg = workload.custom(B=1, H=2, D=D, L=200, dtype=dtype, cfg_id=80)
    layer = arl2.Layer(cfg.B, cfg.H, cfg.L, cfg.D, dtype, device=DEV)
    q, k, v, g = (t.to(DEV) for t in workload.step_inputs(cfg, 0, 0))
    out = torch.empty_like(q)
    layer.denoise_step(q, k, v, g, out=out)
    ref = out.clone()
    torch.cuda.synchronize()
    stream = torch.cuda.Stream()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.stream(stream):
        graph.capture_begin()
        with pytest.raises(RuntimeError):
            stream.synchronize()                       # ends the capture as an invalid one: launches on it are refused
        with pytest.raises(arl2.Arl2Error, match="capture"):
            layer.denoise_step(q, k, v, g, out=out)
        with pytest.raises(RuntimeError):
            graph.capture_end()
    layer.reset()
    out.zero_()
    layer.denoise_step(q, k, v, g, out=out)
    layer.sync_status()
    assert torch.equal(out, ref)
