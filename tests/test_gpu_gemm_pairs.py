"""The projections where the GEMM runs on pairs of CTAs (256 x 256 tiles): row counts around the tile's edges, the ragged
last column tile with the gate logits, and a wait that expires."""
import pytest
import torch

from graph_util import captured_kernels
from paper_2605_16579_b200 import arl2

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _layer(B, H, L, seed):
    d = H * 128
    gen = torch.Generator().manual_seed(seed)
    mk = lambda *s: (torch.randn(*s, generator=gen) / d ** 0.5).to(torch.bfloat16).to(DEV)  # noqa: E731
    w = [mk(d, d), mk(d, d), mk(d, d), mk(d, H), mk(d, d)]
    layer = arl2.Layer(B, H, L, 128, "bf16", device=DEV)
    layer.set_projections(*w)
    return layer, w, torch.randn(B, L, d, generator=gen).to(torch.bfloat16).to(DEV)


def _guarded(shape, dtype):
    """A tensor at the start of a longer one that is filled with NaN."""
    n = 1
    for s in shape:
        n *= s
    whole = torch.full((n + 4096,), float("nan"), dtype=dtype, device=DEV)
    return whole[:n].view(shape), whole[n:]


def _check(got, x, w, bf16):
    # fp32 sums of K products in any order, then one rounding to bf16 (8 significant bits)
    x2, got = x.double().view(-1, x.shape[-1]), got.double().view(-1, w.shape[1])
    ref, mag = x2 @ w.double(), x2.abs() @ w.double().abs()
    bound = x2.shape[1] * 2.0 ** -23 * mag + (2.0 ** -8 * ref.abs() if bf16 else 0.0)
    assert bool(((got - ref).abs() <= bound).all())


def _on_pairs(call):
    """Which of the kernels serves the call (the rule goes by a cost model: a size that it serves otherwise tests nothing here)."""
    (name, grid, _, cluster), = captured_kernels(call)
    pairs = "tc_gemm_pair_kernel" in name
    assert cluster == (2 if pairs else 1) and (not pairs or grid[0] % 2 == 0)
    return pairs


# On pairs: 12 tiles of 256 rows exactly; one whose first CTA has a row and the second none; 48 rows; the second CTA has one
# row; two streams; 5 heads (the gate logits' columns begin in the middle of a tile).  Beside the rule's line: 256 x 256 tiles of one
# CTA, and 128 x 256.
@pytest.mark.parametrize("B,H,L,pairs", [(1, 12, 3072, True), (1, 12, 3073, True), (1, 12, 3120, True), (1, 12, 3201, True),
                                         (2, 12, 1560, True), (1, 5, 6241, True), (1, 12, 1536, False), (1, 12, 1560, False),
                                         (1, 12, 1665, False), (1, 12, 1793, False)])
def test_input_projection_on_pairs(B, H, L, pairs):
    layer, (w_q, w_k, w_v, w_g, _), x = _layer(B, H, L, 31)
    (q, eq), (k, ek), (v, ev) = (_guarded((B, L, H, 128), torch.bfloat16) for _ in range(3))
    g, eg = _guarded((B, L, H), torch.float32)
    assert _on_pairs(lambda: layer.project_in(x, q, k, v, g)) == pairs
    for t in (q, k, v, g):
        t.fill_(float("nan"))
    layer.project_in(x, q, k, v, g)
    layer.sync_status()
    for got, w in ((q, w_q), (k, w_k), (v, w_v)):
        _check(got, x, w, True)
    _check(g, x, w_g, False)
    assert all(bool(torch.isnan(e).all()) for e in (eq, ek, ev, eg))


# whole tiles, and one row in the last tile
@pytest.mark.parametrize("B,L", [(8, 1560), (8, 1536), (1, 12289)])
def test_output_projection_on_pairs(B, L):
    H = 12
    layer, w, o = _layer(B, H, L, 32)
    y, end = _guarded((B, L, H * 128), torch.bfloat16)
    assert _on_pairs(lambda: layer.project_out(o.view(B, L, H, 128), y))
    y.fill_(float("nan"))
    layer.project_out(o.view(B, L, H, 128), y)
    layer.sync_status()
    _check(y, o, w[4], True)
    assert bool(torch.isnan(end).all())


def test_a_wait_that_expires_on_pairs():
    """Every wait at once (0 polls), and at different points of the two CTAs of a pair: they end together, with as many k-blocks
    asked for by one as by the other, and the launches after them are whole."""
    layer, w, x = _layer(1, 12, 3120, 33)
    want = [t.clone() for t in layer.project_in(x)]
    assert _on_pairs(lambda: layer.project_in(x, *[torch.empty_like(t) for t in want]))
    expired = []
    for polls in list(range(17)) * 2:
        layer.debug_set_wait_limit(polls)
        got = layer.project_in(x)
        try:
            layer.sync_status()
            for a, b in zip(got, want):
                assert torch.equal(a, b)
        except arl2.Arl2Error:
            expired.append(polls)
        layer.sync_status()
        layer.debug_set_wait_limit(-1)
        for a, b in zip(layer.project_in(x), want):
            assert torch.equal(a, b)
        layer.sync_status()
    assert expired.count(0) == 2 and len(expired) > 2
