"""The selection in one launch (a cluster, one CTA per block) at the edges of what it takes, against the oracle."""
import threading

import numpy as np
import pytest
import torch

import oracle
from helpers import kernel_names, to_dev_ids
from paper_2607_20457_b200 import binding

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("L,block,chunk,k,sink,vocab,one_launch", [
    (2048, 2048, 2, 5, 3, 31, True),               # one block, 1024 chunks: a thread each
    (2049, 2049, 3, 5, 3, 32, None),               # a token more than a block may have under a score
    (6144, 6144, 8, 5, 3, 33, None),               # as many as it may have without
    (6145, 6145, 8, 5, 3, 33, False),
    (2 * 8192 - 1, 8192, 33, 5, 3, 1000, False),   # as many as the launch of the df table takes
    (2 * 8193 - 1, 8193, 33, 5, 3, 1000, False),
    (2050, 1025, 1, 7, 3, 33, False),              # 1025 chunks
    (16 * 300 - 7, 300, 7, 4, 11, 128256, True),   # 16 blocks, short last chunks, the largest vocabulary
    (17 * 64, 64, 8, 2, 5, 100, False),            # 17 blocks
    (9 * 50 - 49, 50, 3, 17, 50, 1000, True),      # a last block of one token, every chunk selected
    (1024, 128, 33, 3, 0, 5, True),
    (700, 700, 9, 4, 3, 131072, True),             # one block: the vocabulary shared out among CTAs without one; the most entries
    (700, 700, 9, 4, 3, 131073, None),             # of tables for the caller, and one more
    (3 * 500 - 1, 500, 33, 4, 3, 524289, None),    # more entries than the launch of the df table takes
    (2050, 1025, 65, 4, 3, 100, True),             # long chunks in long blocks: the scores that compare positions are apart
    (1024, 1024, 129, 2, 3, 100, True),
])
def test_selection_at_the_edges_of_one_launch(L, block, chunk, k, sink, vocab, one_launch):
    rng = np.random.default_rng(L)
    ids = np.minimum((rng.random(L) ** 3 * vocab).astype(np.uint32), vocab - 1)
    ids_d = to_dev_ids(ids, DEV)
    call = lambda: binding.pulsar_maxidf_select(ids_d, vocab, block, chunk, k, sink, want_df=True, want_idf=True)
    got, ref = call(), oracle.maxidf_select(ids, vocab, block, chunk, k, sink)
    for name in ("sel_chunks", "prefix_idx", "prefix_len"):
        np.testing.assert_array_equal(got[name].cpu().numpy(), ref[name], err_msg=name)
    np.testing.assert_array_equal(got["df"].cpu().numpy().view(np.uint32), ref["df"])
    np.testing.assert_allclose(got["idf"].cpu().numpy(), ref["idf"], rtol=0, atol=1e-6)
    tables = vocab > 131072
    assert (len(kernel_names(call)) == 1) == (one_launch is not False and not tables)
    if one_launch is None and tables:                              # without the tables it is one launch again
        assert len(kernel_names(lambda: binding.pulsar_maxidf_select(ids_d, vocab, block, chunk, k, sink))) == 1
    for mode in binding.SCORE_MODES:
        got = binding.pulsar_chunk_select(ids_d, vocab, block, chunk, k, sink, mode, want_score=True)
        ref = oracle.chunk_select(ids, vocab, block, chunk, k, sink, mode)
        for name in ("sel_chunks", "prefix_idx", "prefix_len"):
            np.testing.assert_array_equal(got[name].cpu().numpy(), ref[name], err_msg=f"{mode} {name}")
        names = kernel_names(lambda: binding.pulsar_chunk_select(ids_d, vocab, block, chunk, k, sink, mode))
        apart = mode == "bm25" and chunk > 64 and block > 1024 or mode == "type_token" and chunk > 128
        one = L <= 16 * block and block <= 2048 and block <= 1024 * chunk and not apart
        table = L <= 16 * block and block <= 8192 and vocab <= 16384 * 32        # the df table in one launch, the scores in theirs
        assert len(names) == (1 if one else 3 if table else 4), names
        assert np.array_equal(got["score"].cpu().numpy(), ref["score"]), mode


@pytest.mark.parametrize("blocks", [4, 17])                       # one launch, and four
def test_threads_with_different_shapes(blocks):
    """The shared memory that a kernel is allowed is the kernel's, not the call's: a small call beside a large one."""
    shapes = [(blocks * 64, 64, vocab) for vocab in (1200000, 500000, 100)] * 5
    failed = []

    def work(L, block, vocab):
        torch.cuda.set_device(0)
        ids = torch.arange(L, dtype=torch.int32, device=DEV) % min(vocab, 97)
        ws = binding._workspace(binding.maxidf_select_workspace_bytes(L, vocab, block, 8, 2, 4), DEV)
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                for _ in range(1500):
                    binding.pulsar_maxidf_select(ids, vocab, block, 8, 2, 4, workspace=ws)
        except Exception as e:
            failed.append((vocab, e))

    threads = [threading.Thread(target=work, args=s) for s in shapes]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert not failed, failed
