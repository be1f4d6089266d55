"""GPU parity: key tiles shared by the two softmax warpgroups, and heads that share query tiles with d = 128."""
import pytest
import torch

from helpers import check_attention
from paper_2607_20457_b200 import binding

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def reference(Q, K, V, causal):
    n, Hq, d = Q.shape
    s = torch.einsum("nhgd,mhd->nhgm", Q.double().view(n, K.shape[1], -1, d), K.double()) / d ** 0.5
    if causal:
        i = torch.arange(n, device=DEV)
        s.masked_fill_((i[None, :] > i[:, None])[:, None, None], float("-inf"))
    O = torch.einsum("nhgm,mhd->nhgd", s.softmax(-1), V.double()).reshape(n, Hq, d)
    return O.cpu().numpy(), s.logsumexp(-1).reshape(n, Hq).cpu().numpy()


def draw(seed, *shapes):
    gen = torch.Generator(device=DEV).manual_seed(seed)
    return [torch.randn(*s, generator=gen, device=DEV, dtype=torch.bfloat16) for s in shapes]


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("L", [1, 63, 64, 65, 128, 129, 192, 193, 400])
def test_key_tiles_whose_second_half_is_short_or_empty(L, d):
    Q, K, V = draw(L, (20, 8, d), (L, 2, d), (L, 2, d))
    Q, K[L // 2] = 3 * Q, 4 * K[L // 2]                          # one key far above the others moves its half's maximum alone
    for n_splits in (1, 0):
        O, LSE = binding.pulsar_phase2_attn(Q, K, V, 1, L, n_splits=n_splits)
        check_attention(O, LSE, *reference(Q, K, V, False), f"L={L}")
    Q, = draw(L + 1, (L, 8, d))
    O, LSE = binding.pulsar_causal_varlen_attn(Q, K, V, [0, L])
    check_attention(O, LSE, *reference(Q, K, V, True), f"causal L={L}")
    assert torch.equal(O, binding.pulsar_causal_varlen_attn(Q, K, V, [0, L])[0])


@pytest.mark.parametrize("g", [2, 4, 8, 16])
def test_heads_share_tiles_of_short_sequences(g):
    """Sequences of 1 to 200 tokens, more pairs of tiles than SMs, d = 128."""
    Hkv, lens = 4, [186, 1, 130, 200, 33, 129, 64, 17] * 5
    cu = [0]
    for n in lens:
        cu.append(cu[-1] + n)
    Q, K, V = draw(g, (cu[-1], g * Hkv, 128), (cu[-1], Hkv, 128), (cu[-1], Hkv, 128))
    O, LSE = binding.pulsar_causal_varlen_attn(Q, K, V, cu)
    for j in list(range(8)) + [len(lens) - 1]:
        r = slice(cu[j], cu[j + 1])
        check_attention(O[r], LSE[r], *reference(Q[r], K[r], V[r], True), f"sequence {j}")
