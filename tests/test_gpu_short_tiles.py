"""GPU parity: key tiles shared by the two softmax warpgroups, and heads that share query tiles with d = 128."""
import pytest
import torch

from helpers import check_attention, kernel_names
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


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("part", [128, 256])
def test_many_short_items_per_sm(part, d):
    """600 and more work items of one or two key tiles, several to an SM: the halves of one item are brought together while
    the next one's are on their way.  Every part has a maximum of its own size, so sums of another item would show."""
    L, nq, Hq, Hkv = part * 300, 20, 8, 2
    Q, K, V = draw(part + d, (nq, Hq, d), (L, Hkv, d), (L, Hkv, d))
    K *= torch.linspace(0.2, 2.0, L // 64, device=DEV).repeat_interleave(64)[torch.randperm(L, device=DEV)][:, None, None].bfloat16()
    want = reference(Q, K, V, False)
    for _ in range(5):
        O, LSE, part_O, part_LSE = binding.pulsar_phase2_attn(Q, K, V, 1, L, n_splits=L // part, want_partials=True)
        check_attention(O, LSE, *want, f"parts of {part}")
    s = torch.einsum("nhgd,jmhd->jnhgm", Q.double().view(nq, Hkv, -1, d), K.double().view(-1, part, Hkv, d)) / d ** 0.5
    assert (part_LSE.double() - s.logsumexp(-1).view(-1, nq, Hq)).abs().max() < 1e-4       # fp32 sums of up to 256 terms
    A = torch.einsum("jnhgm,jmhd->jnhgd", s.softmax(-1), V.double().view(-1, part, Hkv, d)).reshape(part_O.shape)
    assert (part_O.double() - A).abs().max() < 2.0 ** -8 * V.abs().max()       # probabilities in bf16: 2^-9 each, twice that stated


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("Hq,lens", [(8, [128, 256] * 3 + [1400]), (16, [256] * 4 + [1024]), (8, [200] * 3 + [2000])])
def test_short_causal_items_behind_others(Hq, lens, d):
    """One-tile items, more of them than SMs: those of the first sequences, one and two key tiles long, are drawn last."""
    cu = [0]
    for n in lens:
        cu.append(cu[-1] + n)
    Q, K, V = draw(d + Hq, *[(cu[-1], Hq, d)] * 3)
    call = lambda: binding.pulsar_causal_varlen_attn(Q, K, V, cu)
    assert [a for n, a in kernel_names(call) if n == "attn_kernel"] == [[d, 0, 1, 0, 0]]          # one query tile an item
    want = [reference(Q[a:b], K[a:b], V[a:b], True) for a, b in zip(cu, cu[1:])]
    for _ in range(5):
        O, LSE = call()
        for j, (a, b) in enumerate(zip(cu, cu[1:])):
            check_attention(O[a:b], LSE[a:b], *want[j], f"sequence {j}")
