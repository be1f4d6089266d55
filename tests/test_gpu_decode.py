"""GPU parity: queries of at most eight rows per KV head against contexts of 1024 keys or more (csrc/decode.cu)."""
import pytest
import torch

from helpers import check_attention, kernel_names
from paper_2607_20457_b200 import binding

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def reference(Q, K, V, limit):
    """Attention in float64; limit[u]: keys that token u sees."""
    n, Hq, d = Q.shape
    g = Hq // K.shape[1]
    s = torch.einsum("nhgd,mhd->nhgm", Q.double().view(n, -1, g, d), K.double()) / d ** 0.5
    s.masked_fill_((torch.arange(K.shape[0], device=DEV) >= limit[:, None])[:, None, None], float("-inf"))
    O = torch.einsum("nhgm,mhd->nhgd", s.softmax(-1), V.double()).reshape(n, Hq, d)
    return O.cpu().numpy(), s.logsumexp(-1).reshape(n, Hq).cpu().numpy()


def draw(seed, *shapes):
    gen = torch.Generator(device=DEV).manual_seed(seed)
    return [torch.randn(*s, generator=gen, device=DEV, dtype=torch.bfloat16) for s in shapes]


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("L,gen_len,n_new,Hq,Hkv", [
    (1024, 0, 1, 8, 8),            # the shortest context, one row per KV head, an empty shard
    (1025, 15, 2, 8, 2),           # one key past a piece; the shard's pieces end with the new tokens
    (1039, 31, 1, 16, 2),          # eight rows
    (2048, 33, 8, 3, 3),           # eight tokens of one head each: the shard is causal inside its last pieces
    (3001, 500, 2, 4, 1),          # one KV head: a cluster of sixteen CTAs
    (1500, 7, 1, 15, 15),          # fewer CTAs per cluster: 15 and 34 KV heads
    (1100, 1, 1, 34, 34),
    (1030, 3, 1, 200, 200),        # more KV heads than SMs: one CTA each
    (40000, 90, 1, 8, 2),          # long enough for every SM and a merge launch
    (30011, 1000, 4, 2, 1),
    (60000, 5, 1, 16, 16),         # several clusters of four per KV head, fewer than five
])
def test_generation_step(L, gen_len, n_new, Hq, Hkv, d):
    cap = gen_len + n_new + 5
    K, V, Kg, Vg, Q, Kn, Vn = draw(L + Hkv, *[(L, Hkv, d)] * 2, *[(cap, Hkv, d)] * 2, (n_new, Hq, d), *[(n_new, Hkv, d)] * 2)
    Kg[gen_len:], Vg[gen_len:] = float("nan"), float("nan")          # rows that nobody has written yet
    want = Kg.clone(), Vg.clone()
    for t, new in zip(want, (Kn, Vn)):
        t[gen_len: gen_len + n_new] = new
    O, LSE = binding.pulsar_phase2_generate_step(2 * Q, Kn, Vn, K, V, 1, L, Kg, Vg, gen_len)
    for got, w in zip((Kg, Vg), want):
        assert torch.equal(got.view(torch.int16), w.view(torch.int16))
    total = gen_len + n_new
    limit = L + gen_len + 1 + torch.arange(n_new, device=DEV)
    check_attention(O, LSE, *reference(2 * Q, torch.cat([K, Kg[:total]]), torch.cat([V, Vg[:total]]), limit))
    again = binding.pulsar_phase2_generate_step(2 * Q, Kn, Vn, K, V, 1, L, Kg, Vg, gen_len)
    assert torch.equal(O, again[0]) and torch.equal(LSE, again[1])


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("nq,Hq,Hkv,n_splits", [(1, 8, 2, 0), (2, 16, 4, 1), (8, 2, 2, 3), (1, 16, 1, 0)])
def test_query_with_a_late_maximum(nq, Hq, Hkv, n_splits, d):
    """A key far above all others in every warp's range, the later the larger; (1, 16, 1): sixteen rows, which are not taken."""
    L = 5003
    Q, K, V = draw(nq, (nq, Hq, d), (L, Hkv, d), (L, Hkv, d))
    K[::97] *= torch.linspace(1, 6, K[::97].shape[0], device=DEV)[:, None, None].bfloat16()
    call = lambda: binding.pulsar_phase2_attn(Q, K, V, 1, L, n_splits=n_splits)
    O, LSE = call()
    check_attention(O, LSE, *reference(Q, K, V, torch.full((nq,), L, device=DEV)))
    assert ("decode_kernel" in [n for n, _ in kernel_names(call)]) == (nq * Hq // Hkv <= 8)


def test_undefined_keys_show_in_their_rows_only():
    L, Hkv, d = 2000, 2, 128
    Q, K, V = draw(3, (1, 8, d), (L, Hkv, d), (L, Hkv, d))
    want, _ = binding.pulsar_phase2_attn(Q, K, V, 1, L)
    K[1234, 1] = float("nan")
    O, _ = binding.pulsar_phase2_attn(Q, K, V, 1, L)
    assert O[:, 4:].isnan().all() and torch.equal(O[:, :4], want[:, :4])
