"""The step as one call against its three calls."""
import numpy as np
import pytest
import torch

from helpers import kernel_names, to_dev_ids
from paper_2607_20457_b200 import binding
from paper_2607_20457_b200 import workloads as W
from paper_2607_20457_b200.pipeline import ContextEncoder

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("shape", [
    dict(),                                                     # 128 work items: Phase 2 has SMs of its own
    dict(nq=1),                                                 # Phase 2 of few rows, one launch
    dict(nq=300, Hq=8, Hkv=2, d=128),                           # more work items in Phase 2 than SMs
    dict(sink=0, k=0),                                          # no prefix: no gather between
    dict(L=17 * 256, block_size=256, chunk=16, k=2, nq=5),      # 17 blocks: the selection's four launches
    dict(L=4001, block_size=1000, chunk=24, nq=33, Hq=8, Hkv=2, d=128),
    dict(L=1300, block_size=1300, nq=64),                       # one block
])
def test_one_call_equals_three(shape):
    """Two contexts in turn through one encoder: whatever a step leaves in its workspaces and outputs is another context's, or
    not a number, when the next one reads too early."""
    w = W.shrink(W.CONFIGS["tiny"], **shape)
    enc, three = ContextEncoder(w, DEV, slots=6), ContextEncoder(w, DEV)
    gen = torch.Generator(device=DEV).manual_seed(w.L + w.nq)
    inputs, want = [], []
    for seed in range(2):
        Q, K, V = (torch.randn(w.L, h, w.d, generator=gen, device=DEV, dtype=torch.bfloat16) for h in (w.Hq, w.Hkv, w.Hkv))
        Qq = torch.randn(w.nq, w.Hq, w.d, generator=gen, device=DEV, dtype=torch.bfloat16)
        inputs.append((to_dev_ids(ids_with_rare_chunks(w, seed), DEV), Q, K, V, Qq))
        for t in (three.ws_select, three.ws_p1, three.ws_p2):
            t.fill_(0xFF)
        events = [torch.cuda.Event() for _ in range(4)]
        want.append([t.clone() for t in outputs(three.step_device(*inputs[-1], record=events))])
    if w.k and w.n_blocks > 1:                                  # the two select different chunks
        assert not torch.equal(want[0][4], want[1][4]) and not torch.equal(want[0][6], want[1][6])
    for poisoned in (False, True):
        for slot in enc.slots if poisoned else []:
            for t in (slot["O1"], slot["LSE1"], slot["O2"], slot["LSE2"]):
                t.fill_(float("nan"))
            for t in slot["sel"]:
                t.fill_(-0x01010102)
        got = []
        for i, slot in enumerate(enc.slots):                    # back to back: a step beside the end of the one before
            if poisoned:
                for t in (enc.ws_select, enc.ws_p1, enc.ws_p2):
                    t.fill_(0xFF)
            got.append(outputs(enc.step_device(*inputs[i % 2], slot=slot)))
        for i, res in enumerate(got):
            assert all(torch.equal(a, b) for a, b in zip(res, want[i % 2])), (poisoned, i)
    assert int(enc.status.item()) == 0 and int(three.status.item()) == 0


def ids_with_rare_chunks(w, seed):
    """Ids that every block has, and k chunks of each block with an id of their own."""
    rng = np.random.default_rng(seed)
    ids = rng.integers(0, 8, w.L).astype(np.uint32)
    for b in range(w.n_blocks):
        for c in rng.choice(w.chunks_per_block, w.k, replace=False):
            ids[min(b * w.block_size + c * w.chunk, w.L - 1)] = 1000 + b * w.chunks_per_block + c
    return ids


def outputs(r):
    return [r[k] for k in ("O1", "LSE1", "O2", "LSE2", "prefix_idx")] + [r["sel"]["prefix_len"], r["sel"]["sel_chunks"]]


def _encoder(**shape):
    w = W.shrink(W.CONFIGS["tiny"], **shape)
    enc = ContextEncoder(w, DEV)
    Q, K, V = (t.to(DEV) for t in W.qkv(w))
    return w, enc, (to_dev_ids(W.token_ids(w), DEV), Q, K, V, W.phase2_query(w).to(DEV))


def _one_call(w, enc, args, slot, **other):
    ids, Q, K, V, Qq = args
    at = dict(Qq=Qq, O=slot["O1"], LSE=slot["LSE1"], O2=slot["O2"], LSE2=slot["LSE2"], sel=slot["sel"], K=K, V=V,
              ws=(enc.ws_select, enc.ws_p1, enc.ws_p2), ids=ids) | other
    return binding.pulsar_encode_step(at["ids"], w.vocab_size, w.block_size, w.chunk, w.k, w.sink, Q, at["K"], at["V"], at["Qq"], at["sel"],
                                      at["O"], at["LSE"], at["O2"], at["LSE2"], at["ws"], n_splits=enc.n_splits, status=enc.status)


def test_query_and_buffers_are_checked():
    w, enc, args = _encoder(Hq=4, Hkv=2)
    slot = enc.slots[0]
    bf = lambda *s: torch.empty(*s, dtype=torch.bfloat16, device=DEV)
    sel = slot["sel"]
    bad = [(ValueError, dict(Qq=bf(w.nq, 2, w.d))), (ValueError, dict(Qq=bf(w.nq, w.Hq, 2 * w.d))),      # a query of another shape
           (ValueError, dict(O=bf(w.L, w.Hq, w.d - 1))), (ValueError, dict(O2=bf(w.nq - 1, w.Hq, w.d))),
           (ValueError, dict(LSE=slot["LSE1"][1:])), (ValueError, dict(LSE2=slot["LSE2"][1:])),
           (TypeError, dict(O=None)), (TypeError, dict(O2=slot["O2"].float())), (TypeError, dict(LSE=slot["LSE1"].cpu())),
           (TypeError, dict(O=bf(w.L, w.Hq, 2 * w.d)[..., ::2])),
           (ValueError, dict(sel=(sel[0][:w.k], *sel[1:]))), (ValueError, dict(sel=(sel[0], sel[1][:5], sel[2]))),
           (TypeError, dict(ws=(enc.ws_select, enc.ws_p1, None))), (TypeError, dict(ws=(enc.ws_select, enc.ws_p1.cpu(), enc.ws_p2)))]
    before = binding.launch_count()
    for error, other in bad:
        with pytest.raises(error):
            _one_call(w, enc, args, slot, **other)
    assert binding.launch_count() == before
    want = {k: slot[k].clone() for k in ("O1", "O2")} if _one_call(w, enc, args, slot) else None
    _one_call(w, enc, args, slot, LSE=None, LSE2=None)                       # which are wanted or not
    assert all(torch.equal(slot[k], t) for k, t in want.items())


def test_what_one_call_does_not_take_goes_through_three():
    w, enc, args = _encoder(Hq=4, Hkv=2, nq=64)
    full = {k: t.clone() for k, t in enc.step_device(*args).items() if k != "sel"}
    left = {k: None for k in ("O1", "LSE1", "O2", "LSE2", "sel")}            # outputs left to the calls to allocate
    for slot in (left, {**enc.slots[0], "LSE1": None}, {**enc.slots[0], "LSE2": None}):
        got = enc.step_device(*args, slot=slot)
        assert all(torch.equal(got[k], t) for k, t in full.items())
    few = args[4][:, :2].contiguous()                                        # a query of fewer heads than the context's
    got = enc.step_device(*args[:4], few)
    O2, _ = binding.pulsar_phase2_attn(few, args[2], args[3], 1, w.L, n_splits=enc.n_splits)
    assert torch.equal(got["O2"].reshape(-1)[: O2.numel()], O2.reshape(-1))


@pytest.mark.parametrize("nq", [1, 48])
@pytest.mark.parametrize("shared", ["workspaces", "O2 in Q", "LSE2 in the selection's workspace", "Qq in O", "none"])
def test_shared_memory_puts_phase_2_last(shared, nq):
    """What three calls in a row may share, one call may: Phase 2 then follows the other two."""
    w, enc, args = _encoder(nq=nq)
    ids, Q, K, V, Qq = args
    slot = enc.slots[0]
    want = {k: t.clone() for k, t in enc.step_device(*args).items() if k != "sel"}
    one = torch.empty(max(t.numel() for t in (enc.ws_select, enc.ws_p1, enc.ws_p2)), dtype=torch.uint8, device=DEV)
    keep = Q.clone()
    at = dict(workspaces=dict(ws=(one, one, one)), none={})
    at["O2 in Q"] = dict(O2=Q[3: 3 + nq])                                   # Q is used up when Phase 2 writes
    at["LSE2 in the selection's workspace"] = dict(LSE2=enc.ws_select[256: 256 + 4 * nq * w.Hq].view(torch.float32).view(nq, w.Hq))
    at["Qq in O"] = dict(Qq=slot["O1"][:nq])                                # the query is Phase 1's output
    other = at[shared]
    for _ in range(3):
        Q.copy_(keep)
        _one_call(w, enc, args, slot, **other)
        O2, LSE2 = other.get("O2", slot["O2"]).clone(), other.get("LSE2", slot["LSE2"]).clone()
        if shared == "Qq in O":
            ref = binding.pulsar_phase2_attn(want["O1"][:nq].contiguous(), K, V, 1, w.L, n_splits=enc.n_splits)
        else:
            ref = want["O2"], want["LSE2"]
        assert torch.equal(O2, ref[0]) and torch.equal(LSE2, ref[1])
        for k in ("O1", "LSE1", "prefix_idx"):
            assert torch.equal(want[k], slot["sel"][1][: w.prefix_total] if k == "prefix_idx" else slot[k]), k
    Q.copy_(keep)
    names = [n for n, _ in kernel_names(lambda: _one_call(w, enc, args, slot, **other))]
    phase2 = max(i for i, n in enumerate(names) if n in ("attn_kernel", "decode_kernel")) if shared != "none" else names.index("decode_kernel" if nq == 1 else "attn_kernel")
    assert (phase2 > names.index("gather_prefix_kernel")) == (shared != "none"), names
