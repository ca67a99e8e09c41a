"""Upper bounds of what the first cut keeps, from the tokens near the query first: documents with more near tokens than are
collected at a time, masks whose last word is partial, every row width, and both sides of the rule that skips the step."""
import numpy as np
import pytest

from helpers import unit_rows
from test_gpu_batch_scan import check, corpus, queries

pytestmark = pytest.mark.gpu


# D, q_len, centroids, documents, shortest, longest, queries, nprobe, n_prune
CALLS = [
    (32, 32, 1_029, 9_000, 1, 400, 257, 4, 260),         # 32-byte rows
    (32, 64, 2_047, 3_000, 500, 1_500, 220, 1, 300),     # 64-byte rows, hundreds of near tokens
    (64, 90, 999, 3_000, 300, 900, 220, 1, 300),         # 128-byte rows
    (64, 50, 1_500, 6_000, 100, 500, 165, 1, 400),       # ... of other query lengths
    (32, 100, 1_000, 9_000, 20, 90, 330, 2, 200),        # too many near tokens: all rows at once
    (32, 32, 1_029, 9_000, 1, 400, 41, 4, 60),           # too few documents: the same
    (128, 32, 120_003, 20_000, 90, 160, 250, 32, 263),   # 6-bit codes
    (32, 40, 107_001, 9_000, 150, 250, 220, 16, 300),    # ... without a mask
]


@pytest.mark.parametrize("call", CALLS)
def test_kept_candidates_are_bounded_like_the_oracle_orders_them(call):
    arrays = corpus(*call)
    check(arrays, queries(np.random.default_rng(call[1]), arrays[0], call[6], call[1]), call[7], call[8])


@pytest.mark.parametrize("call", CALLS)
def test_the_masks_of_a_scan_by_query_lead_to_the_same_documents(call):
    """Stages 3 to 5 on the table and candidates of the search that the test above checks: the other kernels that write the masks."""
    import torch
    import paper_2608_23553_b200 as pkg
    B, nq, nprobe, n_prune = call[6], call[1], call[7], call[8]
    arrays = corpus(*call)
    gix = pkg.Index(*(torch.from_numpy(a).cuda() for a in arrays), 2)
    q = torch.from_numpy(queries(np.random.default_rng(nq), arrays[0], B, nq)).cuda()
    taps = gix.alloc_taps(B, nq, nprobe, n_prune, ci=False)
    ids, scores = (t.clone() for t in gix.search(q, nprobe, n_prune, 10, taps=taps))
    pruned = taps.pruned.clone()
    got = gix.run_stages(3, 5, q, B, nq, nprobe, n_prune, 10, taps)
    assert gix.status() == 0
    assert torch.equal(taps.pruned, pruned) and torch.equal(got[0], ids) and torch.equal(got[1], scores)


# q_len, query tokens near one direction
@pytest.mark.parametrize("nq,many", [(32, 8), (47, 8), (60, 16), (64, 16), (100, 32)])
def test_bounds_hold_for_query_tokens_of_unlike_thresholds(nq, many):
    """A bound adds up a threshold for every query token without a near document token.  Here `many` neighbouring tokens have high
    thresholds (they lie by a cluster of 40 centroids), four times n_prune documents have a token just below those and match eight or
    more of the other tokens exactly, and documents that repeat one near token take half of the places among the first best: a bound
    that adds up other tokens' thresholds than its own drops documents of the top n_prune."""
    rng = np.random.default_rng(nq)
    D, K, N, B, n_prune = 64, 2_000, 4_000, 328, 200
    long = nq > 64
    high = np.arange(nq // 2, nq // 2 + many)
    row = 32 if nq <= 32 else 64 if nq <= 64 else 128
    # the tokens at the places of the high ones when a row's columns lie in 32 runs of row / 32
    hit = [c for c in high // (row // 32) + 32 * (high % (row // 32)) if c < nq and c not in high] or list(range(8))
    cent = unit_rows(rng, K, D)
    x = unit_rows(rng, 1, D)
    cluster = np.arange(K - 40, K)
    cent[cluster] = x + 0.8 / np.sqrt(D) * rng.standard_normal((40, D))
    cent[cluster] /= np.linalg.norm(cent[cluster], axis=1, keepdims=True)
    below = cluster[np.argsort(cent[cluster] @ x[0])[:20]]
    doclens = rng.integers(200 if long else 100, 301 if long else 201, N).astype(np.int32)
    first = np.concatenate([[0], np.cumsum(doclens)])
    cids = rng.integers(len(hit), K - 40, first[-1]).astype(np.int32)
    docs = rng.permutation(N)
    for t in first[docs[:4 * n_prune]]:
        cids[t:t + len(hit)] = np.arange(len(hit))
        cids[t + len(hit)] = rng.choice(below)
    for t in first[docs[4 * n_prune:4 * n_prune + 180]]:
        cids[t:t + 40] = rng.integers(0, len(hit))
    codes = rng.integers(0, 256, (first[-1], D // 4)).astype(np.uint8)
    q = cent[rng.integers(len(hit), K - 40, (B, nq))] + 0.3 / np.sqrt(D) * rng.standard_normal((B, nq, D))
    q[:, hit] = cent[:len(hit)] + 0.1 / np.sqrt(D) * rng.standard_normal((B, len(hit), D))
    q[:, high] = x + 0.02 / np.sqrt(D) * rng.standard_normal((B, many, D))
    q = (q / np.linalg.norm(q, axis=2, keepdims=True)).astype(np.float32)
    check((cent, cids, codes, doclens), q, 8, n_prune)
