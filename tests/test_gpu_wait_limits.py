"""Waits that expire after some polls, so that the roles of a kernel give up at different points of the work, and some not at
all: the launch ends at once with nothing left in flight, reports the time-out if there was one, and the context then gives
the bits it gave before."""
import time

import pytest
import torch

from paper_2605_16579_b200 import arl2, workload

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
POLLS = (0, 1, 2, 3, 4, 6, 8, 12, 16, 24, 32, 64, 128, 256)


def _layer(cfg, flags=0):
    layer = arl2.Layer(cfg.B, cfg.H, cfg.L, 128, "bf16", device=DEV, flags=flags)
    layer.set_params(*(w.to(DEV) for w in workload.feature_weights(cfg)), *(t.to(DEV) for t in workload.rope_tables(cfg.L, 128)))
    layer.set_state(torch.randn(cfg.B, cfg.H, 128, 128, generator=torch.Generator().manual_seed(9)))
    return layer


def _ended(layer, polls, call):
    """Runs the call under the limit; whether all of its waits ended."""
    layer.debug_set_wait_limit(polls)
    torch.cuda.synchronize()
    begin = time.monotonic()
    call()
    try:
        layer.sync_status()
        ended = True
    except arl2.Arl2Error as e:
        assert "status -4" in str(e)
        ended = False
    assert time.monotonic() - begin < 1.0        # (a pass takes well under a millisecond)
    layer.debug_set_wait_limit(-1)
    assert polls > 0 or not ended
    return ended


# one item per CTA; more items than CTAs
@pytest.mark.parametrize("B,H,L", [(1, 3, 300), (1, 40, 1100)])
@pytest.mark.parametrize("gate", ["head", "channel"])
def test_denoise_pass(B, H, L, gate):
    cfg = workload.custom(B=B, H=H, D=128, L=L, dtype="bf16", cfg_id=191)
    layer = _layer(cfg, arl2.ARL2_FLAG_GATE_ELEMENTWISE if gate == "channel" else 0)
    q, k, v, g = (t.to(DEV) for t in workload.step_inputs(cfg, 0, 0))
    if gate == "channel":
        g = torch.randn(B, L, H, 128, generator=torch.Generator().manual_seed(7)).to(DEV)
    want = layer.denoise_step(q, k, v, g).clone()
    layer.sync_status()
    for polls in POLLS:
        out = torch.full_like(want, float("nan"))
        if _ended(layer, polls, lambda: layer.denoise_step(q, k, v, g, out=out)):
            assert torch.equal(out, want)
        assert torch.equal(layer.denoise_step(q, k, v, g), want)
        layer.sync_status()


@pytest.mark.parametrize("rule", ["gated_linear", "delta"])
def test_commit(rule):
    cfg = workload.custom(B=1, H=5, D=128, L=1500, dtype="bf16", cfg_id=192)
    layer = _layer(cfg)
    k, v, a = (t.to(DEV) for t in workload.commit_inputs(cfg, 0))
    beta = workload.beta_logits(cfg, 0).to(DEV)
    before = layer.get_state()

    def commit():
        if rule == "delta":
            layer.commit_delta(k, v, a, beta)
        else:
            layer.commit(k, v, a)

    commit()
    layer.sync_status()
    after = layer.get_state()
    for polls in POLLS:
        layer.set_state(before)
        ended = _ended(layer, polls, commit)
        assert torch.equal(layer.get_state(), after if ended else before)
        layer.set_state(before)
        commit()
        layer.sync_status()
        assert torch.equal(layer.get_state(), after)


# tiles of one CTA, and of pairs of CTAs
@pytest.mark.parametrize("H,L", [(3, 1000), (12, 1560), (12, 3120)])
def test_input_projection(H, L):
    d = H * 128
    gen = torch.Generator().manual_seed(33)
    mk = lambda *s: (torch.randn(*s, generator=gen) / d ** 0.5).to(torch.bfloat16).to(DEV)  # noqa: E731
    layer = arl2.Layer(1, H, L, 128, "bf16", device=DEV)
    layer.set_projections(mk(d, d), mk(d, d), mk(d, d), mk(d, H), mk(d, d))
    x = torch.randn(1, L, d, generator=gen).to(torch.bfloat16).to(DEV)
    want = [t.clone() for t in layer.project_in(x)]
    layer.sync_status()
    for polls in POLLS:
        got = [torch.empty_like(t) for t in want]
        if _ended(layer, polls, lambda: layer.project_in(x, *got)):
            assert all(torch.equal(a, b) for a, b in zip(got, want))
        assert all(torch.equal(a, b) for a, b in zip(layer.project_in(x), want))
        layer.sync_status()
