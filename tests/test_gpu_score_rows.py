"""The score table for every way its rows are stored (eight tokens at a time, four, one by one) and its tiles end: query-token
rows that fill no tile, end inside a thread's eight or straddle queries, centroids that fill no tile; bit for bit."""
import numpy as np
import pytest
import torch

import oracle
from helpers import random_corpus, unit_rows

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nq,B", [(1, 1), (1, 33), (3, 11), (4, 9), (5, 7), (8, 5), (12, 3), (16, 3), (24, 3), (31, 2), (32, 3),
                                  (33, 2), (40, 3), (47, 1), (64, 2), (101, 2)])
@pytest.mark.parametrize("K", [1, 121, 257])
def test_score_table_equals_oracle(nq, B, K):
    import paper_2608_23553_b200 as pkg
    cent, cids, codes, doclens = random_corpus(K + nq, 20, K, 96, 2)
    gix = pkg.Index(*(torch.from_numpy(a).cuda() for a in (cent, cids, codes, doclens)), 2)
    rng = np.random.default_rng(nq)
    q = np.stack([unit_rows(rng, nq, 96) for _ in range(B)])
    taps = gix.alloc_taps(B, nq, 1, 4)
    gix.run_stages(1, 1, torch.from_numpy(q).cuda(), B, nq, 1, 4, 2, taps)
    assert gix.status() == 0
    table = taps.score_table.cpu().numpy()
    for b in range(B):
        assert np.array_equal(table[b], oracle.score_table(q[b], cent))
