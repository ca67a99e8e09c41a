"""Stage 3's first cut (one number per token) against the oracle: batches and corpora large enough for the library to use
it, all stages of the first and the last query."""
import numpy as np
import pytest
import torch

import oracle
from helpers import random_corpus, unit_rows
from parity import check_query, taps_to_numpy

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("D,nbits,nq,K,N,len_lo,len_hi,B,nprobe,n_prune,shift,copies", [
    (32, 2, 32, 509, 20_000, 1, 80, 260, 1, 300, 0, 1),          # 16-bit numbers from the 8-bit table
    (64, 2, 64, 2_000, 20_001, 20, 61, 256, 1, 1_111, 1, 1),      # two column groups; centroid ids 4 bytes off 16
    (128, 2, 32, 120_003, 9_999, 60, 99, 280, 16, 50, 3, 1),      # 6-bit codes, K not a multiple of five
    (32, 1, 64, 106_497, 5_000, 200, 300, 170, 8, 20, 2, 1),      # ... just above the 16-bit limit
    (96, 1, 21, 700, 20_000, 1, 99, 21, 2, 200, 0, 1),            # exact table, q_len < 32
    (32, 2, 100, 3_000, 12_345, 10, 70, 45, 1, 500, 1, 1),        # ... four column groups
    (32, 2, 40, 107_001, 8_000, 90, 120, 25, 16, 64, 0, 1),       # ... 6-bit codes
    (64, 2, 47, 2_000, 9_000, 20, 90, 60, 1, 300, 0, 1),          # ... rows of an odd number of values, two per lane
    (32, 2, 127, 1_000, 6_000, 20, 70, 80, 1, 200, 0, 1),         # ... four per lane, the longest query
    (64, 2, 32, 6_000, 24_000, 1, 70, 256, 1, 5_900, 0, 1),        # queries with fewer candidates than 1.5 n_prune
    (32, 2, 32, 300, 20_000, 1, 80, 260, 1, 333, 0, 50),          # every document 50 times: masses of equal scores
])
def test_filtered_searches_match_the_oracle(D, nbits, nq, K, N, len_lo, len_hi, B, nprobe, n_prune, shift, copies):
    import paper_2608_23553_b200 as pkg
    cent, cids, codes, doclens = random_corpus(300 + nq + D, N // copies, K, D, nbits, len_lo=len_lo, len_hi=len_hi)
    if copies > 1:
        cids, codes, doclens = (np.concatenate([a] * copies) for a in (cids, codes, doclens))
    oix = oracle.make_index(cent, cids, codes, doclens, nbits)
    padded = torch.zeros(shift + len(cids), dtype=torch.int32, device="cuda")
    padded[shift:] = torch.from_numpy(cids).cuda()
    gix = pkg.Index(torch.from_numpy(cent).cuda(), padded[shift:], torch.from_numpy(codes).cuda(),
                    torch.from_numpy(doclens).cuda(), nbits)
    rng = np.random.default_rng(nq)
    q = cent[rng.integers(0, K, size=(B, nq))] + 0.3 / np.sqrt(D) * rng.standard_normal((B, nq, D)).astype(np.float32)
    q = (q / np.linalg.norm(q, axis=2, keepdims=True)).astype(np.float32)
    k = min(n_prune, 25)
    taps = gix.alloc_taps(B, nq, nprobe, n_prune, table=False)
    ids, sc = gix.search(torch.from_numpy(q).cuda(), nprobe, n_prune, k, taps=taps)
    assert gix.status() == 0
    tn = taps_to_numpy(taps)
    ids, sc = ids.cpu().numpy(), sc.cpu().numpy()
    for b in (0, B - 1):
        res = oracle.pipeline(q[b], oix, nprobe, n_prune, k)
        check_query(tn, b, res, ids[b], sc[b], k, n_prune, table=False)
