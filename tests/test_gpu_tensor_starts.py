"""Output tensors that start on a 16-byte boundary but not on a 32-byte one, and per-channel gate logits that start at any
element, through every tensor-core kernel that writes or reads them: the same bits as from aligned tensors."""
import pytest
import torch

from paper_2605_16579_b200 import arl2, workload

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _shifted(t, elements, odd):
    """A copy of t whose first element lies `elements` behind a 256-byte boundary."""
    buf = torch.full((t.numel() + 256,), float("nan"), dtype=t.dtype, device=DEV)
    v = buf[elements:elements + t.numel()].view(t.shape)
    v.copy_(t)
    assert v.data_ptr() % odd == odd // 2
    return v, buf


# one item per CTA; more items than CTAs; a last wave cut into key ranges; heads walked whole and in runs
@pytest.mark.parametrize("B,H,L", [(1, 3, 300), (1, 40, 1100), (1, 12, 3000), (2, 2, 1030)])
@pytest.mark.parametrize("op", ["denoise", "clean", "token_level", "teacher", "channel_gates"])
def test_same_bits_at_any_start(op, B, H, L):
    cfg = workload.custom(B=B, H=H, D=128, L=L, dtype="bf16", cfg_id=171)
    flags = arl2.ARL2_FLAG_GATE_ELEMENTWISE if op == "channel_gates" else 0
    layer = arl2.Layer(cfg.B, cfg.H, cfg.L, cfg.D, cfg.dtype, device=DEV, flags=flags)
    layer.set_params(*(w.to(DEV) for w in workload.feature_weights(cfg)), *(t.to(DEV) for t in workload.rope_tables(L, 128)))
    layer.reset()
    kc, vc, a = (t.to(DEV) for t in workload.commit_inputs(cfg, 0))
    layer.commit(kc, vc, a)
    before = layer.get_state()
    q, k, v, g = (t.to(DEV) for t in workload.step_inputs(cfg, 1, 0))
    alpha = workload.token_gate_logits(cfg, 1)[0].to(DEV)
    if op == "channel_gates":
        g = torch.randn(B, L, H, 128, generator=torch.Generator().manual_seed(7)).to(DEV)

    def run(gate, out):
        if op == "clean":
            layer.set_state(before)
            return layer.clean_pass(q, kc, vc, gate, a, out=out)
        if op == "token_level":
            return layer.denoise_step_token_level(q, k, v, gate, alpha, out=out)
        if op == "teacher":
            return layer.teacher_step(q, k, v, out=out)
        return layer.denoise_step(q, k, v, gate, out=out)

    ref = run(g, torch.empty_like(q)).clone()
    assert torch.isfinite(ref).all()
    out, buf = _shifted(torch.empty_like(q), 8, 32)      # 16 bytes
    out.fill_(float("nan"))
    gate = _shifted(g, 2, 16)[0] if op == "channel_gates" else g
    run(gate, out)
    layer.sync_status()
    assert torch.equal(out, ref)
    assert torch.isnan(buf[:8]).all() and torch.isnan(buf[8 + out.numel():]).all()
