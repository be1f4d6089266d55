"""GPU parity: causal attention over assembled inputs of different lengths (Algorithm 1 line 8)."""
import numpy as np
import pytest
import torch

import oracle
from helpers import check_attention, kernel_names
from paper_2607_20457_b200 import binding, workloads as W

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def assemble(w, X, pidx, plen):
    """Rows of Input_i = [prefix_i | block_i] for every block, packed back to back (Eq. 4)."""
    parts, cu = [], [0]
    for i in range(w.n_blocks):
        rows = list(pidx[: plen[i]]) + list(range(i * w.block_size, (i + 1) * w.block_size))
        parts.append(X[torch.tensor(rows)])
        cu.append(cu[-1] + len(rows))
    return torch.cat(parts).contiguous(), cu


def test_arbitrary_lengths():
    w = W.shrink(W.CONFIGS["tiny"], L=1500, block_size=1500, Hq=4, Hkv=2, d=128)
    Q, K, V = W.qkv(w, q_scale=2.0)
    cu = [0, 1, 130, 131, 515, 900, 1500]                      # 1 row, ragged tiles, odd and even tile counts
    status = binding.new_status(DEV)
    O, LSE = binding.pulsar_causal_varlen_attn(Q.to(DEV), K.to(DEV), V.to(DEV), cu, status=status)
    torch.cuda.synchronize()
    assert int(status.item()) == 0
    Oref, Lref = oracle.causal_varlen_attn(Q, K, V, cu)
    print(check_attention(O, LSE, Oref, Lref, "varlen"))


def test_assembled_pulsar_inputs_and_agreement_with_the_gathering_operator():
    # At the first layer the prefix keys are the global rows, so the block rows of the assembled
    # run must agree with pulsar_phase1_attn, which gathers the same rows.
    w = W.shrink(W.CONFIGS["tiny"], L=2048, block_size=512, chunk=16, k=4, sink=64, Hq=4, Hkv=1, d=64)
    sel = oracle.maxidf_select(W.needle_ids(w), w.vocab_size, w.block_size, w.chunk, w.k, w.sink)
    pidx, plen = sel["prefix_idx"], sel["prefix_len"]
    Q, K, V = W.qkv(w)
    Qa, cu = assemble(w, Q, pidx, plen)
    Ka, _ = assemble(w, K, pidx, plen)
    Va, _ = assemble(w, V, pidx, plen)
    assert [b - a for a, b in zip(cu[:-1], cu[1:])] == [w.block_size + int(p) for p in plen]   # n_i of Eq. 14
    O, LSE = binding.pulsar_causal_varlen_attn(Qa.to(DEV), Ka.to(DEV), Va.to(DEV), cu)
    Oref, Lref = oracle.causal_varlen_attn(Qa, Ka, Va, cu)
    print(check_attention(O, LSE, Oref, Lref, "assembled"))
    O1, L1, _, _ = binding.pulsar_phase1_attn(Q.to(DEV), K.to(DEV), V.to(DEV), w.block_size,
                                              torch.from_numpy(pidx).to(DEV), torch.from_numpy(plen).to(DEV))
    torch.cuda.synchronize()
    for i in range(w.n_blocks):
        blk = slice(cu[i + 1] - w.block_size, cu[i + 1])
        own = slice(i * w.block_size, (i + 1) * w.block_size)
        assert (O[blk].float() - O1[own].float()).abs().max().item() <= 2e-2
        assert (LSE[blk] - L1[own]).abs().max().item() <= 1e-3


def test_16k_config_assembled_sampled_sequences():
    w = W.CONFIGS["16k"]
    pidx, plen = W.first_k_prefix(w)
    Q, K, V = W.qkv(w)
    Qa, cu = assemble(w, Q, pidx, plen)
    Ka, _ = assemble(w, K, pidx, plen)
    Va, _ = assemble(w, V, pidx, plen)
    O, LSE = binding.pulsar_causal_varlen_attn(Qa.to(DEV), Ka.to(DEV), Va.to(DEV), cu)
    torch.cuda.synchronize()
    # the oracle on the last (longest) sequence, sampled rows
    a, b = cu[-2], cu[-1]
    rows = np.unique(np.concatenate([np.arange(0, 8), np.arange(b - a - 8, b - a),
                                     np.random.default_rng(0).integers(0, b - a, 48)]))
    Oref, Lref = oracle.phase1_attn(Qa[a:b], Ka[a:b], Va[a:b], b - a, np.zeros(0, np.int32), np.zeros(1, np.int32),
                                    rows=rows)
    idx = torch.from_numpy(rows + a).to(DEV)
    print(check_attention(O[idx], LSE[idx], Oref, Lref, "16k assembled, last sequence"))


def test_bad_offsets_are_rejected_on_the_host():
    z = torch.zeros(64, 2, 64, dtype=torch.bfloat16, device=DEV)
    for cu in ([0, 10, 10, 64], [1, 64], [0, 32]):
        with pytest.raises(binding.PulsarError) as e:
            binding.pulsar_causal_varlen_attn(z, z, z, cu)
        assert e.value.status == 2


def test_kv_discard_keeps_each_blocks_own_rows():
    """Appendix F: after the pass over the assembled inputs only the last block_size rows of each are
    kept -- the same rows a boolean mask that is true on the last block_size positions selects --
    and the retained cache is the original K, V (every context token once)."""
    w = W.CONFIGS["tiny"]
    _, K, V = W.qkv(w)
    pidx, plen = W.first_k_prefix(w)
    rows, cu = [], [0]
    for i in range(w.n_blocks):
        rows += list(pidx[: plen[i]]) + list(range(i * w.block_size, (i + 1) * w.block_size))
        cu.append(len(rows))
    idx = torch.tensor(rows)
    Ka, Va = K[idx].contiguous().to(DEV), V[idx].contiguous().to(DEV)
    Kr, Vr = binding.pulsar_retain_block_kv(Ka, Va, cu, w.block_size)
    torch.cuda.synchronize()
    for i in range(w.n_blocks):
        is_bi = torch.zeros(cu[i + 1] - cu[i], dtype=torch.bool)
        is_bi[-w.block_size:] = True
        seg = Ka[cu[i]: cu[i + 1]].cpu()[is_bi]
        assert torch.equal(Kr[i * w.block_size: (i + 1) * w.block_size].cpu(), seg)
    assert torch.equal(Kr.cpu(), K) and torch.equal(Vr.cpu(), V)
    with pytest.raises(binding.PulsarError):
        binding.pulsar_retain_block_kv(Ka, Va, cu, w.block_size + cu[1] + 1)       # longer than the first input


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("n_seq,length", [(1, 1), (2, 129), (36, 300), (37, 300), (3, 1500)])
def test_few_and_many_work_items(n_seq, length, d):
    """Fewer pairs of query tiles than SMs (at most 148): work items of one tile, or of two where that is the shorter time."""
    gen = torch.Generator().manual_seed(n_seq * length)
    lens = [length + 7 * (j % 3) for j in range(n_seq)]
    cu = np.concatenate([[0], np.cumsum(lens)]).astype(np.int32)
    Q = (2 * torch.randn(int(cu[-1]), 2, d, generator=gen)).to(torch.bfloat16)
    K, V = (torch.randn(int(cu[-1]), 1, d, generator=gen).to(torch.bfloat16) for _ in range(2))
    status = binding.new_status(DEV)
    O, LSE = binding.pulsar_causal_varlen_attn(Q.to(DEV), K.to(DEV), V.to(DEV), cu.tolist(), status=status)
    Oref, Lref = oracle.causal_varlen_attn(Q, K, V, cu)
    torch.cuda.synchronize()
    assert int(status.item()) == 0
    check_attention(O, LSE, Oref, Lref, f"{n_seq} x {length} d={d}")


def test_kv_discard_takes_values_in_any_shape():
    """Only K's shape says how many heads of which size a row has; V may come as plain rows."""
    K, V = (torch.randn(300, 2, 64, device=DEV).bfloat16() for _ in range(2))
    Kr, Vr = binding.pulsar_retain_block_kv(K, V, [0, 130, 300], 100)
    K2, V2 = binding.pulsar_retain_block_kv(K, V.view(300, 128), [0, 130, 300], 100)
    assert torch.equal(Kr, K2) and torch.equal(Vr, V2) and torch.equal(Vr[:100], V[30:130])


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("Hq,Hkv,lens", [(2, 1, [300 + 7 * (j % 5) for j in range(60)]),     # one or two key tiles, ragged
                                         (8, 2, [2049, 1000, 3, 1311, 128, 129]), (16, 2, [1500, 777, 1025, 40]),
                                         (6, 2, [2000, 1100, 900, 260])])                    # a group that is not packed
def test_pairs_of_query_tiles(Hq, Hkv, lens, d):
    """More pairs of query tiles than SMs: work items of two tiles, with d = 64 and groups of 2, 4 and 8 heads packed."""
    cu = np.concatenate([[0], np.cumsum(lens)]).astype(np.int32)
    gen = torch.Generator().manual_seed(Hq * len(lens))
    Q = (2 * torch.randn(int(cu[-1]), Hq, d, generator=gen)).to(torch.bfloat16)
    K, V = (torch.randn(int(cu[-1]), Hkv, d, generator=gen).to(torch.bfloat16) for _ in range(2))
    Qd, Kd, Vd = Q.to(DEV), K.to(DEV), V.to(DEV)
    g = Hq // Hkv
    packed = d == 64 and g in (1, 2, 4, 8, 16)
    tokens, heads = (256 // g, Hkv) if packed else (256, Hq)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    repeat = sms // (heads * sum(-(-n // tokens) for n in lens)) + 1                 # as often as it takes
    if repeat > 1:
        lens = lens * repeat
        cu = np.concatenate([[0], np.cumsum(lens)]).astype(np.int32)
        Q, K, V = (x.repeat(repeat, 1, 1) for x in (Q, K, V))
        Qd, Kd, Vd = (x.repeat(repeat, 1, 1) for x in (Qd, Kd, Vd))
    assert len(lens) <= 64 and heads * sum(-(-n // tokens) for n in lens) > sms
    status = binding.new_status(DEV)
    call = lambda: binding.pulsar_causal_varlen_attn(Qd, Kd, Vd, cu.tolist(), status=status)
    O, LSE = call()
    assert [args[:3] for name, args in kernel_names(call) if name == "attn_kernel"] == [[d, 0, 0]]
    Oref, Lref = oracle.causal_varlen_attn(Q, K, V, cu)
    torch.cuda.synchronize()
    assert int(status.item()) == 0
    check_attention(O, LSE, Oref, Lref, f"Hq={Hq} Hkv={Hkv} d={d} {len(lens)} sequences")
