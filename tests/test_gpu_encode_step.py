"""The step as one call against its three calls."""
import pytest
import torch

from helpers import to_dev_ids
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
    w = W.shrink(W.CONFIGS["tiny"], **shape)
    enc = ContextEncoder(w, DEV)
    Q, K, V = (t.to(DEV) for t in W.qkv(w))
    args = to_dev_ids(W.token_ids(w), DEV), Q, K, V, W.phase2_query(w).to(DEV)
    events = [torch.cuda.Event() for _ in range(4)]
    keep = lambda r: [r[k].clone() for k in ("O1", "LSE1", "O2", "LSE2", "prefix_idx")] + [r["sel"]["prefix_len"].clone(), r["sel"]["sel_chunks"].clone()]
    want = keep(enc.step_device(*args, record=events))
    for _ in range(3):                                          # back to back: a step beside the end of the one before
        for t in enc.slots[0].values():
            if isinstance(t, torch.Tensor) and t.dtype == torch.float32:
                t.fill_(7.0)
        got = keep(enc.step_device(*args))
        assert all(torch.equal(a, b) for a, b in zip(got, want))
    assert int(enc.status.item()) == 0
