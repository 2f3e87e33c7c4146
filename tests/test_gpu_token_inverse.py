"""The chunk inverse of arl2_commit_tokens is computed in fp32: its small entries come out of cancelling sums."""
import numpy as np
import pytest
import torch

from paper_2605_16579_b200 import arl2

pytestmark = pytest.mark.gpu

# Keys of 60 common entries of 1/8 and one entry of 1/4 of their own: unit length, the same inner product 15/16
# between any two, every value exact in bf16 (as are the normalised rows).  With rates b_i near 1 the inverse of
# I + diag(b) strictly_lower(K K^T) falls off by 1 - 15/16 b per step away from the diagonal, out of sums whose terms
# are near 1.  The own entry of token i is a row of S of its own, the value vectors are unit vectors: S[64 + i, j] = T_ij b_j / 4.
D, C = 128, 64


def _keys():
    k = torch.zeros(C, D)
    k[:, :60] = torch.where(torch.arange(60) % 3 == 0, -0.125, 0.125)
    k[torch.arange(C), 64 + torch.arange(C)] = 0.25
    return k


@pytest.mark.parametrize("chunk", [0, 1])
@pytest.mark.parametrize("decayed", [False, True])
def test_small_entries_of_the_chunk_inverse(oracle, chunk, decayed):
    B, H, L = 1, 3, 2 * C
    gen = torch.Generator().manual_seed(11 + chunk)
    k, v = torch.zeros(B, L, H, D), torch.zeros(B, L, H, D)
    beta = torch.full((B, L, H), -200.0)              # the other chunk's tokens write nothing
    rows = slice(chunk * C, (chunk + 1) * C)
    k[:] = _keys().repeat(2, 1)[None, :, None, :]
    v[0, rows] = torch.eye(D)[:C, None, :]
    beta[0, rows] = torch.rand(C, H, generator=gen) * 3.0 + 3.0
    k, v = k.bfloat16(), v.bfloat16()
    flags = arl2.ARL2_FLAG_TOKEN_GATES | (arl2.ARL2_FLAG_DELTA_DECAYED_PREDICTION if decayed else 0)
    layer = arl2.Layer(B, H, L, D, "bf16", device="cuda:0", flags=flags)
    layer.set_params()
    layer.commit_tokens(k.cuda(), v.cuda(), None, beta.cuda())
    layer.sync_status()
    got = layer.get_state().double().numpy()[:, :, 64:, :C]
    ref = oracle.commit_tokens(k, v, np.zeros((B, H, D, D)), None, beta, decayed_prediction=decayed)[:, :, 64:, :C]
    # relative: T, diag(b) V' and the product of both are each rounded to bf16, 8 significant bits, so by up to 2^-8 each.
    # absolute, on T (a quarter of it in S): A21 T11 and T22 (.) sum terms that fall off geometrically, so a handful of
    # fp32 roundings of numbers up to 1 in each, with column sums of T up to 2: 8 x 2^-24.  Operands of 16 bits
    # miss it by a factor of 6 and more (3e-6 to 2e-5 on these inputs).
    bound = 3.1 * 2.0 ** -8 * np.abs(ref) + 0.25 * 8 * 2.0 ** -24
    lower = np.tril(np.ones((C, C), dtype=bool), -1)
    small = lower & (np.abs(ref) < 2.0 ** -12)
    assert small.sum() > 1000
    worst = (np.abs(got - ref) / bound)[:, :, lower].max()
    assert worst <= 1.0, f"an entry is off by {worst:.2f} of its bound"
