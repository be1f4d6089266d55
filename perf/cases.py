"""The work that users of this library have it do, as cases to time.

Six kinds of pass, each through the public entry points a program calls:

``step``       one layer of one context: selection, Phase-1 attention, Phase-2 attention of the query
               (``ContextEncoder.step_device``, the repository's headline workload)
``generate``   one generation step of a decoding loop: new tokens appended to the generation shard, then
               attending to the whole context and the shard (``pulsar_phase2_generate_step``)
``query``      another query against a context that is already encoded (``pulsar_phase2_attn``)
``assembled``  one layer over assembled inputs, as the paper's whole-model pass runs it: rotary embedding at the
               inputs' position ids, causal attention inside every input, KV discard
``select``     chunk selection alone, under one of the other chunk scores (``pulsar_chunk_select``)
``rank``       what one GPU runs between its collectives when the blocks of a context are spread over several
               (``ShardedContextEncoder``): selection, packing, Phase 1 and its partial of Phase 2

Inputs: token ids of a Zipf law (s = 1.1) over the vocabulary, Q, K, V ~ N(0,1) in bf16, as everywhere in this
repository.  Sizes come from ``workloads.CONFIGS`` and from ranges around them.
"""
import math

import torch

from paper_2607_20457_b200 import binding
from paper_2607_20457_b200.pipeline import ContextEncoder
from paper_2607_20457_b200.sharding import ShardedContextEncoder, ShardLayout
from paper_2607_20457_b200.workloads import CONFIGS, Workload

DEV = "cuda"
SHAPE = ("L", "block_size", "chunk", "k", "sink", "vocab_size", "Hq", "Hkv", "d")


def _config(name):
    w = CONFIGS[name]
    return {f: getattr(w, f) for f in SHAPE}


def listed():
    return [
        # The smallest context of the configurations: every kernel is short, latency and launches are what is paid.
        dict(name="step_4k", kind="step", **_config("tiny"), nq=32),
        # A short document with a question of 64 tokens.
        dict(name="step_16k", kind="step", **_config("16k"), nq=64),
        # A document as long as it happens to be: nothing divides anything, head dimension 64, a short last block.
        dict(name="step_45k_ragged_d64", kind="step", L=45011, block_size=5000, chunk=30, k=9, sink=50, vocab_size=32000,
             Hq=16, Hkv=4, d=64, nq=37),
        # A long document, 8 blocks of 8192.
        dict(name="step_64k", kind="step", **_config("64k"), nq=128),
        # The headline: 128K tokens in 16 blocks, 8 queries of 64 tokens.
        dict(name="step_128k", kind="step", **_config("128k"), nq=512),
        # Decoding token by token after a short context: the smallest call a decoding loop makes.
        dict(name="generate_1_at_6k", kind="generate", L=6001, n_new=1, gen_len=33, Hq=8, Hkv=2, d=128),
        # Decoding token by token after the longest context: the keys and values stream from HBM.
        dict(name="generate_1_at_128k", kind="generate", L=131072, n_new=1, gen_len=200, Hq=32, Hkv=8, d=128),
        # Several tokens at once (a drafted continuation) after an ordinary context.
        dict(name="generate_12_at_32k", kind="generate", L=32768, n_new=12, gen_len=77, Hq=32, Hkv=8, d=128),
        # A question of 50 tokens against an encoded context of ragged length.
        dict(name="query_50_at_100k", kind="query", L=100003, nq=50, Hq=32, Hkv=8, d=128),
        # One layer of the whole-model pass over the assembled inputs of a 32K context.
        dict(name="assembled_32k", kind="assembled", **_config("32k")),
        # Selection by BM25 over a long context.
        dict(name="select_bm25_128k", kind="select", L=131072, block_size=8192, chunk=32, k=16, sink=64, vocab_size=128256,
             score="bm25"),
        # One of four GPUs that share a 128K context.
        dict(name="rank_of_4_128k", kind="rank", **_config("128k"), n_hosts=4, rank=1, nq=64),
    ]


HEADS = ((4, 1), (8, 2), (16, 4), (32, 8), (8, 8), (16, 2))


def _log_int(rng, lo, hi):
    return max(lo, min(hi, round(math.exp(rng.uniform(math.log(lo), math.log(hi))))))


def _context(rng, longest, whole_blocks=0):
    """A context of 2 to 16 blocks; ``whole_blocks``: its length is a multiple of that many whole blocks."""
    L = _log_int(rng, 2048, longest)
    n_blocks = rng.randint(max(2, -(-L // 8192)), 16)
    block = -(-L // n_blocks)
    chunk = rng.choice((16, 24, 32, 32, 48, 64, rng.randint(15, 64)))
    if rng.random() < 0.4:                                   # lengths that divide, as in the configurations
        block = max(block // 256 * 256, 256)
        chunk = rng.choice((16, 32, 64))
        L = block * -(-L // block)
    if whole_blocks:
        chunk = rng.choice((16, 32, 64))
        block = max(block // chunk * chunk, 256)
        n_blocks = max(whole_blocks, n_blocks // whole_blocks * whole_blocks)
        L = block * n_blocks
    k = rng.randint(1, max(1, min(512, block // 4) // chunk))
    Hq, Hkv = rng.choice(HEADS)
    return dict(L=L, block_size=block, chunk=chunk, k=k, sink=rng.choice((0, 16, 64, rng.randint(1, 64))),
                vocab_size=rng.choice((32000, 50257, 128256)), Hq=Hq, Hkv=Hkv, d=rng.choice((64, 128, 128)))


def draw(rng):
    kind = rng.choices(("step", "generate", "query", "assembled", "select", "rank"), (8, 5, 3, 3, 2, 2))[0]
    if kind == "step":
        return dict(kind=kind, **_context(rng, 120000), nq=_log_int(rng, 1, 512))
    if kind == "generate":
        Hq, Hkv = rng.choice(HEADS)
        return dict(kind=kind, L=_log_int(rng, 2048, 131072), n_new=rng.choice((1, 1, 1, rng.randint(2, 32))),
                    gen_len=rng.randint(0, 1000), Hq=Hq, Hkv=Hkv, d=rng.choice((64, 128, 128)))
    if kind == "query":
        Hq, Hkv = rng.choice(HEADS)
        return dict(kind=kind, L=_log_int(rng, 2048, 131072), nq=_log_int(rng, 1, 512), Hq=Hq, Hkv=Hkv,
                    d=rng.choice((64, 128, 128)))
    if kind == "assembled":
        return dict(kind=kind, **_context(rng, 65536, whole_blocks=1))
    if kind == "select":
        c = _context(rng, 120000)
        return dict(kind=kind, **{f: c[f] for f in ("L", "block_size", "chunk", "k", "sink", "vocab_size")},
                    score=rng.choice(("tf_idf", "bm25", "type_token")))
    n_hosts = rng.choice((2, 4, 8))
    return dict(kind=kind, **_context(rng, 100000, whole_blocks=n_hosts), n_hosts=n_hosts, rank=rng.randrange(n_hosts),
                nq=_log_int(rng, 1, 512))


# ---- inputs ---------------------------------------------------------------------------------------------------------

def _randn(gen, *shape):
    return torch.randn(shape, generator=gen, device=DEV, dtype=torch.bfloat16)


def _ids(gen, L, vocab_size):
    p = torch.arange(1, vocab_size + 1, device=DEV, dtype=torch.float64).pow_(-1.1)
    cdf = p.cumsum(0) / p.sum()
    u = torch.rand(L, generator=gen, device=DEV, dtype=torch.float64)
    return torch.searchsorted(cdf, u, right=True).clamp_(max=vocab_size - 1).to(torch.int32)


def _workload(c, nq=1):
    return Workload(name=c.get("name", "drawn"), nq=nq, **{f: c[f] for f in SHAPE})


def _cu_seqlens(c):
    B, sigma = c["L"] // c["block_size"], c["k"] * c["chunk"]
    cu = [0]
    for i in range(B):
        cu.append(cu[-1] + c["block_size"] + (c["sink"] + i * sigma if i else 0))
    return cu


def prepare(case, seed):
    c, gen = dict(case), torch.Generator(device=DEV).manual_seed(seed)
    kind = c["kind"]
    if kind == "step":
        w = _workload(c, c["nq"])
        return dict(kind=kind, enc=ContextEncoder(w, DEV), ids=_ids(gen, w.L, w.vocab_size),
                    Q=_randn(gen, w.L, w.Hq, w.d), K=_randn(gen, w.L, w.Hkv, w.d), V=_randn(gen, w.L, w.Hkv, w.d),
                    Qq=_randn(gen, w.nq, w.Hq, w.d))
    if kind == "generate":
        L, n, Hq, Hkv, d = c["L"], c["n_new"], c["Hq"], c["Hkv"], c["d"]
        capacity = 1024 + 64                                 # rows the generation shard can grow to
        splits = binding.phase2_choose_splits(n, 1, L, Hq, Hkv, d)
        ws = binding.load_library().pulsar_phase2_generate_workspace_bytes(n, 1, L, Hq, Hkv, d, splits)
        return dict(kind=kind, L=L, gen_len=c["gen_len"], splits=splits, ws=torch.empty(ws, dtype=torch.uint8, device=DEV),
                    Q=_randn(gen, n, Hq, d), Kn=_randn(gen, n, Hkv, d), Vn=_randn(gen, n, Hkv, d),
                    K=_randn(gen, L, Hkv, d), V=_randn(gen, L, Hkv, d),
                    Kg=_randn(gen, capacity, Hkv, d), Vg=_randn(gen, capacity, Hkv, d))
    if kind == "query":
        L, nq, Hq, Hkv, d = c["L"], c["nq"], c["Hq"], c["Hkv"], c["d"]
        return dict(kind=kind, L=L, Q=_randn(gen, nq, Hq, d), K=_randn(gen, L, Hkv, d), V=_randn(gen, L, Hkv, d))
    if kind == "assembled":
        # Selection and the position ids are made once per context; the pass is what every layer repeats.
        cu, ids = _cu_seqlens(c), _ids(gen, c["L"], c["vocab_size"])
        sel = binding.pulsar_maxidf_select(ids, c["vocab_size"], c["block_size"], c["chunk"], c["k"], c["sink"])
        pos = binding.pulsar_assemble_positions(sel["prefix_idx"], sel["prefix_len"], c["L"] // c["block_size"],
                                                c["block_size"], cu[-1], "sparse")
        T, Hq, Hkv, d = cu[-1], c["Hq"], c["Hkv"], c["d"]
        return dict(kind=kind, cu=cu, pos=pos, block_size=c["block_size"], Q=_randn(gen, T, Hq, d),
                    K=_randn(gen, T, Hkv, d), V=_randn(gen, T, Hkv, d))
    if kind == "select":
        return dict(kind=kind, case=c, ids=_ids(gen, c["L"], c["vocab_size"]))
    lay = ShardLayout.make(c["L"] // c["block_size"], c["n_hosts"], c["block_size"], c["chunk"], c["k"], c["sink"])
    Hq, Hkv, d = c["Hq"], c["Hkv"], c["d"]
    rows = lay.n_local * lay.block_size
    enc = ShardedContextEncoder(lay, c["rank"], Hq, Hkv, d, c["vocab_size"], DEV, nq=c["nq"])
    return dict(kind=kind, enc=enc, ids=_ids(gen, c["L"], c["vocab_size"]), Q=_randn(gen, rows, Hq, d),
                K=_randn(gen, rows, Hkv, d), V=_randn(gen, rows, Hkv, d), Qq=_randn(gen, c["nq"], Hq, d),
                # what the all-gather of the ranks' summaries brings
                gathered=_randn(gen, lay.n_hosts, 2, lay.send_rows, Hkv, d))


# ---- one pass -------------------------------------------------------------------------------------------------------

def run(s):
    kind = s["kind"]
    if kind == "step":
        r = s["enc"].step_device(s["ids"], s["Q"], s["K"], s["V"], s["Qq"])
        return dict(O1=r["O1"], LSE1=r["LSE1"], O2=r["O2"], LSE2=r["LSE2"], sel_chunks=r["sel"]["sel_chunks"],
                    prefix_idx=r["sel"]["prefix_idx"], prefix_len=r["sel"]["prefix_len"])
    if kind == "generate":
        O, LSE = binding.pulsar_phase2_generate_step(s["Q"], s["Kn"], s["Vn"], s["K"], s["V"], 1, s["L"], s["Kg"], s["Vg"],
                                                     s["gen_len"], n_splits=s["splits"], workspace=s["ws"])
        return dict(O=O, LSE=LSE, Kg=s["Kg"], Vg=s["Vg"])
    if kind == "query":
        O, LSE = binding.pulsar_phase2_attn(s["Q"], s["K"], s["V"], 1, s["L"])
        return dict(O=O, LSE=LSE)
    if kind == "assembled":
        Q, K = binding.pulsar_rope_apply_qk(s["Q"], s["K"], s["pos"])
        O, LSE = binding.pulsar_causal_varlen_attn(Q, K, s["V"], s["cu"])
        K_ret, V_ret = binding.pulsar_retain_block_kv(K, s["V"], s["cu"], s["block_size"])
        return dict(O=O, LSE=LSE, K_ret=K_ret, V_ret=V_ret)
    if kind == "select":
        c = s["case"]
        return binding.pulsar_chunk_select(s["ids"], c["vocab_size"], c["block_size"], c["chunk"], c["k"], c["sink"],
                                           c["score"], want_score=True)
    enc = s["enc"]
    sel = enc.select(s["ids"])
    send = enc.phase1_pack(s["K"], s["V"])
    O, LSE = enc.phase1_finish(s["gathered"], s["Q"], s["K"], s["V"])
    part = enc.phase2_local(s["Qq"], s["K"], s["V"])
    return dict(sel_chunks=sel["sel_chunks"], prefix_idx=sel["prefix_idx"], send=send, O=O, LSE=LSE, partial=part)


# ---- what a pass cannot do without --------------------------------------------------------------------------------

def _select_bytes(c):
    B = -(-c["L"] // c["block_size"])
    return 4 * (c["L"] + 2 * B * c["k"] * c["chunk"])


def work(case):
    c, kind = dict(case), case["kind"]
    if kind == "select":
        B, C = -(-c["L"] // c["block_size"]), -(-c["block_size"] // c["chunk"])
        return dict(bytes=_select_bytes(c) + 8 * B * C, flops=2 * c["L"])
    Hq, Hkv, d = c["Hq"], c["Hkv"], c["d"]
    row_q, row_kv = 2 * Hq * d, 2 * Hkv * d                  # bytes of one token's Q (or O) and K (or V)
    if kind in ("generate", "query"):
        n = c["n_new"] if kind == "generate" else c["nq"]
        keys = c["L"] + (c["gen_len"] + n if kind == "generate" else 0)
        new = 4 * n * row_kv if kind == "generate" else 0    # KV(q) of the new tokens: read, and written to the shard
        return dict(bytes=2 * keys * row_kv + n * (2 * row_q + 4 * Hq) + new, flops=4 * d * Hq * n * keys)
    L, nb, sigma = c["L"], c["block_size"], c["k"] * c["chunk"]
    if kind == "assembled":
        cu = _cu_seqlens(c)
        T, kept = cu[-1], 2 * L * row_kv
        pairs = sum(n * (n + 1) // 2 for n in (b - a for a, b in zip(cu, cu[1:])))
        return dict(bytes=T * (2 * row_q + 2 * row_kv + 4 * Hq + 4) + kept, flops=4 * d * Hq * pairs + 6 * T * (Hq + Hkv) * d)
    B = -(-L // nb)
    if kind == "step":
        blocks, rows, extra = range(B), L, 0
    else:
        blocks = ShardLayout.make(B, c["n_hosts"], nb, c["chunk"], c["k"], c["sink"]).local_blocks(c["rank"])
        rows = len(blocks) * nb
        # the prefix rows that arrive, the summary rows that leave, the float32 partial instead of bf16
        extra = 2 * row_kv * (c["sink"] + (B - 1) * sigma) + 4 * row_kv * (c["sink"] + len(blocks) * sigma) + c["nq"] * row_q
    pairs = 0
    for i in blocks:
        n = min(nb, L - i * nb)
        pairs += n * (c["sink"] + i * sigma if i else 0) + n * (n + 1) // 2
    nq = c["nq"]
    return dict(bytes=_select_bytes(c) + rows * (2 * row_q + 2 * row_kv + 4 * Hq) + nq * (2 * row_q + 4 * Hq) + extra,
                flops=4 * d * Hq * (pairs + nq * rows))


def tolerance(case):
    # Selection and its scores are the same bit for bit.  The attention outputs are bf16 (half an ulp is 2^-9 of the
    # value) of fp32 sums over probabilities that are themselves rounded to bf16: against the same path in float64 they
    # are off by 2.2e-3 in the norm and by up to 0.04 of max(rms, |value|); four times that is stated.
    return "exact" if case["kind"] == "select" else {"rel": 1e-2, "max": 0.16}
