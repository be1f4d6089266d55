"""GPU parity of the sharded path (block-to-host mapping, Appendix J; Phase-2 exchange, Appendix H).

One GPU: the H ranks run one after the other in this process and the all-gather is a concatenation
of their send buffers (no kernel waits on another).  The sharded result is compared with the
oracle and, row for row, with the unsharded entry points."""
import numpy as np
import pytest
import torch

import oracle
from helpers import check_attention, kernel_names, to_dev_ids
from paper_2607_20457_b200 import binding, cost_model as cm, workloads as W
from paper_2607_20457_b200.sharding import ShardLayout, ShardedContextEncoder

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def make_ranks(w, H, kind):
    lay = ShardLayout.make(w.n_blocks, H, w.block_size, w.chunk, w.k, w.sink, kind)
    return lay, [ShardedContextEncoder(lay, h, w.Hq, w.Hkv, w.d, w.vocab_size, DEV) for h in range(H)]


def sharded_phase1(w, H, kind, ids, Q, K, V):
    lay, ranks = make_ranks(w, H, kind)
    dev_ids = to_dev_ids(ids, DEV)
    local = []
    for h, r in enumerate(ranks):
        rows = torch.from_numpy(lay.local_token_rows(h)).to(DEV)
        local.append((Q[rows].contiguous(), K[rows].contiguous(), V[rows].contiguous(), rows))
        r.select(dev_ids)
    sends = [r.phase1_pack(l[1], l[2]).clone() for r, l in zip(ranks, local)]
    gathered = torch.stack(sends)                                  # what all_gather returns on every rank
    O = torch.empty_like(Q)
    LSE = torch.empty((w.L, w.Hq), dtype=torch.float32, device=DEV)
    for r, (q, k, v, rows) in zip(ranks, local):
        o, lse = r.phase1_finish(gathered, q, k, v)
        O[rows] = o
        LSE[rows] = lse
    torch.cuda.synchronize()
    assert all(int(r.status.item()) == 0 for r in ranks)
    return O, LSE


@pytest.mark.parametrize("kind", cm.MAPPINGS)
@pytest.mark.parametrize("H", [1, 2, 4])
def test_phase1_sharded_equals_unsharded(H, kind):
    w = W.CONFIGS["tiny"]
    ids = W.needle_ids(w)
    Q, K, V = (t.to(DEV) for t in W.qkv(w))
    O, LSE = sharded_phase1(w, H, kind, ids, Q, K, V)
    sel = binding.pulsar_maxidf_select(to_dev_ids(ids, DEV), w.vocab_size, w.block_size, w.chunk, w.k, w.sink)
    O1, LSE1, _, _ = binding.pulsar_phase1_attn(Q, K, V, w.block_size, sel["prefix_idx"], sel["prefix_len"])
    torch.cuda.synchronize()
    assert torch.equal(O, O1) and torch.equal(LSE, LSE1)            # same kernel, same key order
    ref = oracle.maxidf_select(ids, w.vocab_size, w.block_size, w.chunk, w.k, w.sink)
    O_ref, LSE_ref = oracle.phase1_attn(Q.cpu(), K.cpu(), V.cpu(), w.block_size, ref["prefix_idx"], ref["prefix_len"])
    check_attention(O, LSE, O_ref, LSE_ref, f"sharded phase 1 H={H} {kind}")


def test_phase1_sharded_16k_sampled_rows():
    w = W.CONFIGS["16k"]
    ids = W.needle_ids(w)
    Q, K, V = (t.to(DEV) for t in W.qkv(w))
    O, LSE = sharded_phase1(w, 4, "zigzag", ids, Q, K, V)
    ref = oracle.maxidf_select(ids, w.vocab_size, w.block_size, w.chunk, w.k, w.sink)
    rows = W.sample_rows(w, per_block=6)
    O_ref, LSE_ref = oracle.phase1_attn(Q.cpu(), K.cpu(), V.cpu(), w.block_size, ref["prefix_idx"], ref["prefix_len"],
                                        rows=rows)
    r = torch.from_numpy(np.asarray(rows)).to(DEV)
    check_attention(O[r], LSE[r], O_ref, LSE_ref, "sharded phase 1, 16k")


@pytest.mark.parametrize("H,kind", [(1, "contiguous"), (2, "zigzag"), (4, "round_robin"), (4, "zigzag")])
@pytest.mark.parametrize("nq", [1, 37, 512])
def test_phase2_sharded(H, kind, nq):
    w = W.CONFIGS["tiny"]
    _, K, V = (t.to(DEV) for t in W.qkv(w))
    Qq = W.phase2_query(w)
    Qq = (Qq[:nq] if nq <= Qq.shape[0] else Qq.repeat((nq + Qq.shape[0] - 1) // Qq.shape[0], 1, 1)[:nq]).to(DEV)
    Qq = Qq.contiguous()
    lay, ranks = make_ranks(w, H, kind)
    sends = []
    for h, r in enumerate(ranks):
        rows = torch.from_numpy(lay.local_token_rows(h)).to(DEV)
        sends.append(r.phase2_local(Qq, K[rows].contiguous(), V[rows].contiguous()))
    gathered = torch.stack(sends)
    outs = [r.phase2_finish(gathered, nq) for r in ranks]
    torch.cuda.synchronize()
    assert all(int(r.status.item()) == 0 for r in ranks)
    for o, lse in outs[1:]:                                          # every rank ends with the same result
        assert torch.equal(o, outs[0][0]) and torch.equal(lse, outs[0][1])
    O_ref, LSE_ref = oracle.phase2_attn(Qq.cpu(), K.cpu(), V.cpu(), w.n_blocks, w.block_size)
    check_attention(outs[0][0], outs[0][1], O_ref, LSE_ref, f"sharded phase 2 H={H} {kind} nq={nq}")


def test_strided_merge_float32_partial_matches_oracle():
    rng = np.random.default_rng(3)
    J, rows, d, stride = 5, 77, 64, 77 * 64 + 77 + 3 + 16
    stride = (stride + 3) // 4 * 4
    buf = torch.zeros(J * stride, dtype=torch.float32)
    pO = rng.standard_normal((J, rows, d))
    pL = rng.standard_normal((J, rows)) * 4
    pL[2, :5] = -np.inf
    for j in range(J):
        buf[j * stride: j * stride + rows * d] = torch.from_numpy(pO[j].reshape(-1)).float()
        buf[j * stride + rows * d: j * stride + rows * d + rows] = torch.from_numpy(pL[j]).float()
    buf = buf.to(DEV)
    out = torch.empty((rows, d), dtype=torch.float32, device=DEV)
    lse = torch.empty(rows, dtype=torch.float32, device=DEV)
    binding.pulsar_lse_merge_strided(buf, buf[rows * d:], J, stride, stride, rows, d, out, lse)
    O_ref, L_ref = oracle.lse_merge(pO.astype(np.float32).astype(np.float64), pL.astype(np.float32).astype(np.float64))
    assert np.abs(out.cpu().numpy() - O_ref).max() < 2e-6 * max(1.0, np.abs(O_ref).max())
    assert np.abs(lse.cpu().numpy() - L_ref).max() < 1e-5
    with pytest.raises(binding.PulsarError):
        binding.pulsar_lse_merge_strided(buf, buf[rows * d:], J, rows * d - 4, stride, rows, d, out, lse)


def test_gather_rows_and_bad_index():
    K = torch.randn(300, 2, 64, device=DEV).bfloat16()
    V = torch.randn(300, 2, 64, device=DEV).bfloat16()
    idx = torch.tensor([5, 0, 299, 5, 17], dtype=torch.int32, device=DEV)
    Ko, Vo = torch.empty(5, 2, 64, device=DEV, dtype=torch.bfloat16), torch.empty(5, 2, 64, device=DEV, dtype=torch.bfloat16)
    st = binding.new_status(DEV)
    binding.pulsar_gather_kv_rows(K, V, idx, Ko, Vo, status=st)
    assert torch.equal(Ko, K[idx.long()]) and torch.equal(Vo, V[idx.long()]) and int(st.item()) == 0
    idx[2] = 300
    binding.pulsar_gather_kv_rows(K, V, idx, Ko, Vo, status=st)
    assert int(st.item()) & 0x2 and torch.equal(Ko[2], K[0])


@pytest.mark.parametrize("rows,Hkv,d", [(1, 1, 8), (1023, 1, 8), (1025, 1, 8), (341, 3, 8), (342, 3, 8), (9, 16, 128), (700, 5, 24), (4, 1, 9000)])
def test_row_copies_where_rows_and_ctas_do_not_meet(rows, Hkv, d):
    """1024 vectors of 8 elements to a CTA: rows of 1 to 1125 of them, the last CTA full, over and short; one bad index."""
    gen = torch.Generator(device=DEV).manual_seed(rows)
    K, V = (torch.randn(2 * rows + 8, Hkv, d, generator=gen, device=DEV).bfloat16() for _ in range(2))
    idx = torch.randint(0, K.shape[0], (rows,), generator=gen, device=DEV, dtype=torch.int32)
    Ko, Vo = torch.full((2, rows + 1, Hkv, d), 7.0, device=DEV, dtype=torch.bfloat16)
    st = binding.new_status(DEV)
    binding.pulsar_gather_kv_rows(K, V, idx, Ko[:rows], Vo[:rows], status=st)
    assert torch.equal(Ko[:rows], K[idx.long()]) and torch.equal(Vo[:rows], V[idx.long()]) and int(st.item()) == 0
    assert (Ko[rows:] == 7).all() and (Vo[rows:] == 7).all()
    idx[rows // 2] = -1
    binding.pulsar_gather_kv_rows(K, V, idx, Ko[:rows], Vo[:rows], status=st)
    assert int(st.item()) & 0x2 and torch.equal(Ko[:rows], K[idx.clamp(min=0).long()]) and (Vo[rows:] == 7).all()
    # packing: two blocks of `rows` tokens in chunks of one, all but one chunk of each selected in descending order, three sink rows
    n, k, sink = 2, max(rows - 1, 1), min(3, rows)
    sel = torch.arange(rows - 1, rows - 1 - k, -1, device=DEV, dtype=torch.int32).repeat(4, 1)
    Ks, Vs = torch.full((2, sink + n * k + 1, Hkv, d), 7.0, device=DEV, dtype=torch.bfloat16)
    st.zero_()
    binding.pulsar_pack_summary_kv(K[: n * rows], V[: n * rows], rows, sel, torch.tensor([1, 3], dtype=torch.int32, device=DEV), 4, 1, k,
                                   sink, Ks, Vs, status=st)
    src = torch.cat([torch.arange(sink, device=DEV)] + [s * rows + sel[0].long() for s in range(n)])
    assert torch.equal(Ks[:-1], K[src]) and torch.equal(Vs[:-1], V[src]) and int(st.item()) == 0
    assert (Ks[-1] == 7).all() and (Vs[-1] == 7).all()


@pytest.mark.parametrize("H,nq", [(1, 5), (2, 37), (4, 1), (4, 130)])
def test_phase2_with_the_exchange_fused_into_the_merge(H, nq):
    """Every rank merges its slice of the rows straight from all ranks' partial buffers (here all on
    one GPU, addressed through a pointer table as peer memory would be)."""
    from paper_2607_20457_b200.sharding import LocalPeers
    w = W.CONFIGS["tiny"]
    _, K, V = (t.to(DEV) for t in W.qkv(w))
    Qq = W.phase2_query(w)
    Qq = Qq.repeat((nq + Qq.shape[0] - 1) // Qq.shape[0], 1, 1)[:nq].contiguous().to(DEV)
    lay, ranks = make_ranks(w, H, "zigzag")
    peers = LocalPeers(H)
    for h, r in enumerate(ranks):
        rows = torch.from_numpy(lay.local_token_rows(h)).to(DEV)
        r.phase2_local_into(peers, Qq, K[rows].contiguous(), V[rows].contiguous())
    n_rows = nq * w.Hq
    O = torch.empty((n_rows, w.d), dtype=torch.bfloat16, device=DEV)
    LSE = torch.empty(n_rows, dtype=torch.float32, device=DEV)
    covered = 0
    for r in ranks:
        o, lse, begin = r.phase2_merge_slice(peers, nq)
        O[begin: begin + o.shape[0]] = o
        LSE[begin: begin + o.shape[0]] = lse
        covered += o.shape[0]
    torch.cuda.synchronize()
    assert covered == n_rows
    O_ref, LSE_ref = oracle.phase2_attn(Qq.cpu(), K.cpu(), V.cpu(), w.n_blocks, w.block_size)
    check_attention(O.view(nq, w.Hq, w.d), LSE.view(nq, w.Hq), O_ref, LSE_ref, f"fused exchange H={H} nq={nq}")
    # and it is the all-gather path's result exactly (same parts, same order)
    sends = torch.stack([p.clone() for p in peers.buffers])
    O2, LSE2 = ranks[0].phase2_finish(sends, nq)
    assert torch.equal(O2.view(n_rows, w.d), O) and torch.equal(LSE2.view(n_rows), LSE)


_SYMM_WORLD1 = r"""
import os, sys, torch, torch.distributed as dist
os.environ.update(MASTER_ADDR="127.0.0.1", MASTER_PORT=str(29650 + os.getpid() % 200), RANK="0", WORLD_SIZE="1")
torch.cuda.set_device(0)
dist.init_process_group("nccl", device_id=torch.device("cuda", 0))
from paper_2607_20457_b200 import binding, workloads as W
from paper_2607_20457_b200.sharding import ShardLayout, ShardedContextEncoder, SymmetricMemoryPeers, TorchCollective
w = W.CONFIGS["tiny"]
_, K, V = (t.cuda() for t in W.qkv(w))
Qq = W.phase2_query(w).cuda()
lay = ShardLayout.make(w.n_blocks, 1, w.block_size, w.chunk, w.k, w.sink, "zigzag")
enc = ShardedContextEncoder(lay, 0, w.Hq, w.Hkv, w.d, w.vocab_size, "cuda:0", TorchCollective())
peers = SymmetricMemoryPeers()
O, LSE = enc.phase2_fused(peers, Qq, K, V)
O2, LSE2 = enc.phase2(Qq, K, V)                      # NCCL all-gather path at world size 1
O1, LSE1 = binding.pulsar_phase2_attn(Qq, K, V, w.n_blocks, w.block_size)
torch.cuda.synchronize()
assert torch.equal(O, O2) and torch.equal(LSE, LSE2)
assert (O.float() - O1.float()).abs().max().item() < 1e-2 and (LSE - LSE1).abs().max().item() < 1e-3
assert int(enc.status.item()) == 0
dist.destroy_process_group()
print("SYMM-OK")
"""


def test_symmetric_memory_and_nccl_plumbing_at_world_size_one():
    """The rendezvous, the device-side barrier and the NCCL all-gather as one rank (the only
    multi-process configuration a single GPU allows)."""
    import os, subprocess, sys
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    env = dict(os.environ, PYTHONPATH=root + os.pathsep + os.environ.get("PYTHONPATH", ""))
    out = subprocess.run([sys.executable, "-c", _SYMM_WORLD1], capture_output=True, text=True, timeout=600, env=env,
                         cwd=root)
    assert out.returncode == 0 and "SYMM-OK" in out.stdout, (out.stdout + out.stderr)[-3000:]


def test_phase1_sharded_at_the_128k_configuration_equals_the_unsharded_call():
    """Eight ranks with two blocks each (zigzag), run in turn: bit-identical to pulsar_phase1_attn, whose
    output at this configuration is checked against the oracle in test_gpu_phase1.py."""
    w = W.CONFIGS["128k"]
    ids = W.token_ids(w)
    Q, K, V = (t.to(DEV) for t in W.qkv(w))
    O, LSE = sharded_phase1(w, 8, "zigzag", ids, Q, K, V)
    sel = binding.pulsar_maxidf_select(to_dev_ids(ids, DEV), w.vocab_size, w.block_size, w.chunk, w.k, w.sink)
    O1, LSE1, _, _ = binding.pulsar_phase1_attn(Q, K, V, w.block_size, sel["prefix_idx"], sel["prefix_len"])
    torch.cuda.synchronize()
    assert torch.equal(O, O1) and torch.equal(LSE, LSE1)


def form_of(fn):
    """Query tiles per work item (1 or 2) of the attention launch in ``fn``: the third template argument of the kernel."""
    found = [args for name, args in kernel_names(fn) if name == "attn_kernel"]
    assert len(found) == 1
    return 1 if found[0][2] else 2


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("B,block,Hq,prefix,form", [
    (1, 1024, 32, 0, 1),          # 128 pairs, tiles that differ by up to a factor of eight
    (1, 1024, 32, 8192, 2),       # the same behind a long prefix: all alike (d = 64: 110 us in pairs, 130 us in tiles)
    (1, 512, 32, 8192, 1),        # 64 pairs: every tile has an SM of its own
    (8, 512, 8, 7168, 1),         # a prefix that grows from block to block (d = 64: 61 us in tiles, 95 us in pairs)
    (4, 1024, 32, 3072, 2),       # 512 pairs
])
def test_form_follows_the_time_that_the_items_take(B, block, Hq, prefix, form, d):
    if torch.cuda.get_device_properties(0).multi_processor_count != 148:
        pytest.skip("the shapes are those of 148 SMs")
    Hkv = Hq // 4
    gen = torch.Generator(device=DEV).manual_seed(B * block + prefix)
    rnd = lambda n, h: torch.randn(n, h, d, generator=gen, device=DEV, dtype=torch.bfloat16)
    L = B * block
    Q, K, V = rnd(L, Hq), rnd(L, Hkv), rnd(L, Hkv)
    Kp, Vp = (rnd(prefix, Hkv), rnd(prefix, Hkv)) if prefix else (None, None)
    plen = torch.tensor([prefix * i // (B - 1) if B > 1 else prefix for i in range(B)], dtype=torch.int32, device=DEV)
    O, LSE = binding.pulsar_phase1_attn_sharded(Q, K, V, block, Kp, Vp, plen)
    assert form_of(lambda: binding.pulsar_phase1_attn_sharded(Q, K, V, block, Kp, Vp, plen)) == form
    for i in (0, B - 1):
        for h in (0, Hq - 1):
            rows, n = slice(i * block, (i + 1) * block), int(plen[i])
            k, v = K[rows, h // 4].double(), V[rows, h // 4].double()
            if n:
                k, v = torch.cat([Kp[:n, h // 4].double(), k]), torch.cat([Vp[:n, h // 4].double(), v])
            x = Q[rows, h].double() @ k.T / d ** 0.5
            x.masked_fill_(torch.arange(n + block, device=DEV) > n + torch.arange(block, device=DEV)[:, None], float("-inf"))
            l = x.logsumexp(1)
            check_attention(O[rows, h: h + 1], LSE[rows, h: h + 1], ((x - l[:, None]).exp() @ v)[:, None].cpu().numpy(),
                            l[:, None].cpu().numpy(), f"block {i} head {h}")


def test_form_of_assembled_inputs():
    if torch.cuda.get_device_properties(0).multi_processor_count != 148:
        pytest.skip("the shapes are those of 148 SMs")
    for n_seq, length, Hq, form in ((1, 4096, 8, 1), (4, 1024, 8, 2), (16, 300, 8, 2), (2, 1024, 8, 1)):
        cu = [i * length for i in range(n_seq + 1)]
        Q, K = (torch.zeros(cu[-1], h, 64, dtype=torch.bfloat16, device=DEV) for h in (Hq, Hq // 4))
        assert form_of(lambda: binding.pulsar_causal_varlen_attn(Q, K, K, cu)) == form, (n_seq, length, Hq)
