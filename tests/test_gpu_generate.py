"""GPU parity: the Phase-2 generation step against the oracle (Algorithm 1 lines 11-16)."""
import numpy as np
import pytest
import torch

import oracle
from helpers import check_attention
from paper_2607_20457_b200 import binding, workloads as W

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def run_steps(w, steps, cap, q_scale=1.0, n_splits=0, shard_fill=0.0):
    _, K, V = W.qkv(w)
    Kd, Vd = K.to(DEV), V.to(DEV)
    gen = torch.Generator().manual_seed(21)
    Kgen_o = np.zeros((cap, w.Hkv, w.d), np.uint16); Vgen_o = np.zeros_like(Kgen_o)
    Kgen_d = torch.full((cap, w.Hkv, w.d), shard_fill, dtype=torch.bfloat16, device=DEV); Vgen_d = Kgen_d.clone()
    status = binding.new_status(DEV)
    gen_len = 0
    for n_new in steps:
        Qn = (torch.randn(n_new, w.Hq, w.d, generator=gen) * q_scale).to(torch.bfloat16)
        Kn = torch.randn(n_new, w.Hkv, w.d, generator=gen).to(torch.bfloat16)
        Vn = torch.randn(n_new, w.Hkv, w.d, generator=gen).to(torch.bfloat16)
        O, LSE = binding.pulsar_phase2_generate_step(Qn.to(DEV), Kn.to(DEV), Vn.to(DEV), Kd, Vd, w.n_blocks,
                                                     w.block_size, Kgen_d, Vgen_d, gen_len, n_splits=n_splits,
                                                     status=status)
        Oref, Lref = oracle.generate_step(Qn, Kn, Vn, K, V, Kgen_o, Vgen_o, gen_len)
        torch.cuda.synchronize()
        assert int(status.item()) == 0
        print(check_attention(O, LSE, Oref, Lref, f"{w.name} step n_new={n_new} gen_len={gen_len}"))
        gen_len += n_new
        # the shard on the device holds the same bits as the oracle's
        got = Kgen_d[:gen_len].cpu().view(torch.int16).numpy().view(np.uint16)
        np.testing.assert_array_equal(got, Kgen_o[:gen_len])
    return gen_len


def test_tiny_config_query_then_tokens():
    run_steps(W.CONFIGS["tiny"], [32, 1, 1, 1, 7], cap=64)


def test_shard_longer_than_one_key_tile_and_peaked_logits():
    # 150 + 140 rows: the shard spans three key tiles, the new tokens two query tiles
    w = W.shrink(W.CONFIGS["tiny"], L=2048, block_size=512, Hq=8, Hkv=2, d=128)
    run_steps(w, [150, 140, 1], cap=320, q_scale=3.0, n_splits=4)


def test_unwritten_shard_rows_may_hold_anything():
    """The rows of the generation shard past the live ones belong to nobody yet (a cache taken from
    an uninitialised allocation): filled with NaN they must not reach the result, neither while the
    shard is shorter than one key tile nor when its last tile is partial."""
    w = W.shrink(W.CONFIGS["tiny"], L=2048, block_size=512, Hq=8, Hkv=2, d=128)
    run_steps(w, [5, 1, 130, 1], cap=512, shard_fill=float("nan"))
    run_steps(W.CONFIGS["tiny"], [1, 1], cap=200, shard_fill=float("nan"))


def test_16k_config_query_of_64_then_decode():
    run_steps(W.CONFIGS["16k"], [64, 1, 1], cap=128)


def test_capacity_is_checked_on_the_host():
    w = W.CONFIGS["tiny"]
    _, K, V = W.qkv(w)
    z = lambda n, h: torch.zeros(n, h, w.d, dtype=torch.bfloat16, device=DEV)
    with pytest.raises(binding.PulsarError) as e:
        binding.pulsar_phase2_generate_step(z(4, w.Hq), z(4, w.Hkv), z(4, w.Hkv), K.to(DEV), V.to(DEV), w.n_blocks,
                                            w.block_size, z(8, w.Hkv), z(8, w.Hkv), gen_len=6)
    assert e.value.status == 2


def test_step_captured_as_a_cuda_graph_replays_to_the_same_results():
    """One generation step (append, attention started beside it, merge started beside the attention)
    recorded as a CUDA graph: the replay equals the call-by-call step bit for bit, also after the
    inputs in the captured buffers have changed."""
    w = W.CONFIGS["tiny"]
    _, K, V = W.qkv(w)
    Kd, Vd = K.to(DEV), V.to(DEV)
    gen = torch.Generator().manual_seed(5)
    cap, gen_len, n_new = 64, 9, 1
    rnd = lambda n, h: torch.randn(n, h, w.d, generator=gen).to(torch.bfloat16).to(DEV)
    Kgen, Vgen = rnd(cap, w.Hkv), rnd(cap, w.Hkv)
    Qn, Kn, Vn = rnd(n_new, w.Hq), rnd(n_new, w.Hkv), rnd(n_new, w.Hkv)
    status = binding.new_status(DEV)
    n_splits = binding.phase2_choose_splits(n_new, w.n_blocks, w.block_size, w.Hq, w.Hkv, w.d)
    ws = binding._workspace(binding.load_library().pulsar_phase2_generate_workspace_bytes(
        n_new, w.n_blocks, w.block_size, w.Hq, w.Hkv, w.d, n_splits), DEV)
    O = torch.empty_like(Qn)

    def step():
        return binding.pulsar_phase2_generate_step(Qn, Kn, Vn, Kd, Vd, w.n_blocks, w.block_size, Kgen, Vgen, gen_len,
                                                   n_splits=n_splits, out=O, workspace=ws, status=status)

    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):
        step()
    torch.cuda.current_stream().wait_stream(side)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        _, LSE_g = step()
    for fresh in (False, True):
        if fresh:                                       # new token in the captured buffers
            Qn.copy_(rnd(n_new, w.Hq)); Kn.copy_(rnd(n_new, w.Hkv)); Vn.copy_(rnd(n_new, w.Hkv))
        O.zero_(); LSE_g.zero_()
        graph.replay()
        torch.cuda.synchronize()
        O_replay, LSE_replay, K_row = O.clone(), LSE_g.clone(), Kgen[gen_len].clone()
        _, LSE_e = step()
        torch.cuda.synchronize()
        assert torch.equal(O_replay, O) and torch.equal(LSE_replay, LSE_e)
        assert torch.equal(K_row, Kn[0]) and torch.equal(Kgen[gen_len], Kn[0])
        to_np = lambda t: t.cpu().view(torch.int16).numpy().view(np.uint16)
        Oref, Lref = oracle.generate_step(Qn.cpu(), Kn.cpu(), Vn.cpu(), K, V, to_np(Kgen).copy(), to_np(Vgen).copy(),
                                          gen_len)
        print(check_attention(O_replay, LSE_replay, Oref, Lref, f"graph replay fresh={fresh}"))
    assert int(status.item()) == 0


@pytest.mark.parametrize("n_new", [1, 3, 9, 32, 33])
@pytest.mark.parametrize("L,gen_len,n_splits", [(1, 0, 1), (128, 127, 1), (129, 128, 2), (1000, 700, 3), (300, 900, 2), (2049, 5, 17), (640, 0, 5)])
def test_shard_beside_the_last_part_of_the_context(L, gen_len, n_splits, n_new):
    """The shard shares the last context part, or has a part of its own when the others hold the whole context; its new
    rows are appended by the attention kernel (one query tile) or by a launch before it (33 tokens of 4 heads)."""
    Hq, Hkv, d = 8, 2, 64
    gen = torch.Generator().manual_seed(L + gen_len + n_new)
    K, V = (torch.randn(L, Hkv, d, generator=gen).to(torch.bfloat16) for _ in range(2))
    cap = gen_len + n_new + 3
    Kg, Vg = (torch.randn(cap, Hkv, d, generator=gen).to(torch.bfloat16) for _ in range(2))
    Qn = (2 * torch.randn(n_new, Hq, d, generator=gen)).to(torch.bfloat16)
    Kn, Vn = (torch.randn(n_new, Hkv, d, generator=gen).to(torch.bfloat16) for _ in range(2))
    Kg_d, Vg_d = Kg.to(DEV), Vg.to(DEV)
    status = binding.new_status(DEV)
    O, LSE = binding.pulsar_phase2_generate_step(Qn.to(DEV), Kn.to(DEV), Vn.to(DEV), K.to(DEV), V.to(DEV), 1, L, Kg_d, Vg_d,
                                                 gen_len, n_splits=n_splits, status=status)
    Kg_o, Vg_o = (x.view(torch.int16).numpy().view(np.uint16).copy() for x in (Kg, Vg))
    Oref, Lref = oracle.generate_step(Qn, Kn, Vn, K, V, Kg_o, Vg_o, gen_len)
    torch.cuda.synchronize()
    assert int(status.item()) == 0
    check_attention(O, LSE, Oref, Lref, f"L={L} gen_len={gen_len} parts={n_splits} n_new={n_new}")
    for got, want in ((Kg_d, Kg_o), (Vg_d, Vg_o)):             # the rows beyond the new ones stay as they were
        np.testing.assert_array_equal(got.cpu().view(torch.int16).numpy().view(np.uint16), want)


@pytest.mark.parametrize("L,n_new,gen_len,Hq,Hkv", [(6001, 1, 33, 8, 2), (4416, 1, 58, 16, 4), (3271, 1, 642, 8, 2),
                                                    (6314, 1, 163, 16, 2), (4416, 12, 77, 8, 2), (2500, 64, 200, 16, 4)])
def test_parts_longer_than_the_contexts_cost_no_accuracy(L, n_new, gen_len, Hq, Hkv):
    """Where context and shard are cut together the parts are longer than n_splits parts of the context alone (two key tiles
    instead of one here).  P's rounding error is smallest in short parts (the largest probability of a part's first
    key tile is exactly 1): formed with a maximum that lags behind, P is 8-10 % further from float64 with two tiles
    (4-5 % with more than 32 query rows, two estimates of 16,000 outputs or more, each good to 1 %)."""
    d, dev = 128, DEV
    tiles = lambda n: (n + 127) // 128
    n_splits = binding.phase2_choose_splits(n_new, 1, L, Hq, Hkv, d)
    assert n_splits == tiles(L)
    gen = torch.Generator(device=dev).manual_seed(L)
    rnd = lambda n, h: torch.randn(n, h, d, generator=gen, device=dev, dtype=torch.bfloat16)
    err = torch.zeros(2, dtype=torch.float64, device=dev)
    for _ in range(max(4, 16 // n_new)):
        K, V, Kg, Vg = rnd(L, Hkv), rnd(L, Hkv), rnd(gen_len + n_new, Hkv), rnd(gen_len + n_new, Hkv)
        Q, Kn, Vn = rnd(n_new, Hq), rnd(n_new, Hkv), rnd(n_new, Hkv)
        O, _ = binding.pulsar_phase2_generate_step(Q, Kn, Vn, K, V, 1, L, Kg, Vg, gen_len)
        Kc, Vc = torch.cat([K, Kg]), torch.cat([V, Vg])          # the shard has its new rows by now
        n = Kc.shape[0]
        O2, _ = binding.pulsar_phase2_attn(Q, Kc, Vc, 1, n, n_splits=tiles(n))
        s = torch.einsum("nhgd,mhd->nhgm", Q.view(n_new, Hkv, Hq // Hkv, d).double(), Kc.double()) / d ** 0.5
        later = torch.arange(n, device=dev) > L + gen_len + torch.arange(n_new, device=dev)[:, None]
        ref = lambda s: torch.einsum("nhgm,mhd->nhgd", s.softmax(-1), Vc.double()).reshape(n_new, Hq, d)
        refs = ref(s.masked_fill(later[:, None, None], float("-inf"))), ref(s)
        err += torch.stack([(x.double() - r).square().sum() for x, r in zip((O, O2), refs)])
    a, b = err.sqrt().tolist()
    assert a <= 1.025 * b, (a, b)


@pytest.mark.parametrize("d,n_new,launches", [(128, 1, 2), (128, 2, 2), (128, 3, 2), (128, 17, 2), (128, 32, 2), (128, 33, 3),
                                              (128, 100, 3), (64, 4, 2), (64, 5, 2), (64, 64, 2), (64, 65, 3)])
def test_rows_are_appended_by_the_attention_kernel_or_before_it(d, n_new, launches):
    """One warp appends the new rows of its KV head, 512 vectors of 16 bytes at most; more come from a launch of their own."""
    L, gen_len, H = 700, 61, 2
    gen = torch.Generator().manual_seed(d + n_new)
    rnd = lambda n: torch.randn(n, H, d, generator=gen).to(torch.bfloat16)
    K, V, Kg, Vg, Qn, Kn, Vn = rnd(L), rnd(L), rnd(gen_len + n_new + 2), rnd(gen_len + n_new + 2), rnd(n_new), rnd(n_new), rnd(n_new)
    Kg_d, Vg_d = Kg.to(DEV), Vg.to(DEV)
    args = [t.to(DEV) for t in (Qn, Kn, Vn, K, V)]
    before = binding.launch_count()
    O, LSE = binding.pulsar_phase2_generate_step(*args, 1, L, Kg_d, Vg_d, gen_len)
    assert binding.launch_count() - before == launches
    Kg_o, Vg_o = (x.view(torch.int16).numpy().view(np.uint16).copy() for x in (Kg, Vg))
    Oref, Lref = oracle.generate_step(Qn, Kn, Vn, K, V, Kg_o, Vg_o, gen_len)
    check_attention(O, LSE, Oref, Lref, f"d={d} n_new={n_new}")
    for got, want in ((Kg_d, Kg_o), (Vg_d, Vg_o)):
        np.testing.assert_array_equal(got.cpu().view(torch.int16).numpy().view(np.uint16), want)
