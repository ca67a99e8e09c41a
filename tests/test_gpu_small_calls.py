"""The kernels that small calls take (probes by column, short-chunk compaction, shared-memory bitmaps) at the edges of their
ranges, against the oracle."""
import numpy as np
import pytest
import torch

import oracle
from helpers import random_corpus, unit_rows
from parity import check_query, taps_to_numpy

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("K,N,nq,nprobe,B", [
    (1, 33, 5, 1, 1),               # one centroid, one chunk of two words
    (1_023, 2_048, 32, 32, 1),      # one warp per column, not quite full; exactly one chunk
    (1_025, 2_049, 33, 4, 2),       # a second warp with one row; a chunk with one word
    (4_000, 70_000, 13, 7, 3),
    (31_000, 9_000, 2, 3, 4),       # 31 warps per column
    (300, 524_289, 4, 2, 2),        # one document past the short chunks: counted chunks
    (64, 12_000, 16, 2, 40),        # a batch whose lists set every word often (shared-memory bitmap, one block per query)
])
def test_small_calls_match_the_oracle(K, N, nq, nprobe, B):
    import paper_2608_23553_b200 as pkg
    D, nbits, n_prune, k = 32, 2, 20, 7
    cent, cids, codes, doclens = random_corpus(K + N, N, K, D, nbits, len_lo=1, len_hi=3)
    oix = oracle.make_index(cent, cids, codes, doclens, nbits)
    gix = pkg.Index(*(torch.from_numpy(a).cuda() for a in (cent, cids, codes, doclens)), nbits)
    rng = np.random.default_rng(7)
    q = np.stack([unit_rows(rng, nq, D) for _ in range(B)])
    taps = gix.alloc_taps(B, nq, nprobe, n_prune, table=False)
    ids, sc = gix.search(torch.from_numpy(q).cuda(), nprobe, n_prune, k, taps=taps)
    assert gix.status() == 0
    tn = taps_to_numpy(taps)
    ids, sc = ids.cpu().numpy(), sc.cpu().numpy()
    for b in sorted({0, B - 1}):
        check_query(tn, b, oracle.pipeline(q[b], oix, nprobe, n_prune, k), ids[b], sc[b], k, n_prune, table=False)
