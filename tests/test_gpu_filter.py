"""Stage 3's first cut (one number per token) against the oracle: batches and corpora large enough for the library to use
it, all stages of the first and the last query."""
import numpy as np
import pytest
import torch

import oracle
from helpers import random_corpus, unit_rows
from parity import check_query, taps_to_numpy

pytestmark = pytest.mark.gpu


# cut: whether the call runs it (the last four rows have too many centroids, or too long a pruning list, for what their
# candidates hold).  The two before those scan one query at a time, the others all queries together.
CALLS = [
    (1, 32, 2, 32, 509, 20_000, 1, 80, 260, 1, 300, 0, 1),          # 16-bit numbers from the 8-bit table
    (1, 64, 2, 64, 2_000, 20_001, 20, 61, 256, 1, 1_111, 1, 1),      # two column groups; centroid ids 4 bytes off 16
    (1, 128, 2, 32, 120_003, 30_000, 60, 99, 250, 32, 50, 3, 1),     # 6-bit codes, K not a multiple of five
    (1, 32, 1, 64, 106_497, 9_000, 200, 300, 170, 16, 20, 2, 1),     # ... just above the 16-bit limit
    (1, 96, 1, 21, 700, 20_000, 1, 99, 21, 2, 200, 0, 1),            # exact table, q_len < 32
    (1, 32, 2, 100, 3_000, 12_345, 10, 70, 45, 1, 500, 1, 1),        # ... four column groups
    (1, 32, 2, 40, 107_001, 16_000, 90, 120, 25, 32, 64, 0, 1),      # ... 6-bit codes
    (1, 64, 2, 47, 2_000, 9_000, 20, 90, 60, 1, 300, 0, 1),          # ... rows of an odd number of values, two per lane
    (1, 32, 2, 127, 1_000, 6_000, 20, 70, 80, 1, 200, 0, 1),         # ... four per lane, the longest query
    (1, 32, 2, 32, 300, 20_000, 1, 80, 260, 1, 333, 0, 50),          # every document 50 times: masses of equal scores
    (1, 64, 2, 32, 12_000, 60_000, 30, 50, 260, 1, 100, 1, 1),
    (1, 96, 1, 21, 8_000, 40_000, 1, 99, 260, 1, 100, 3, 1),
    (0, 128, 2, 32, 120_003, 9_999, 60, 99, 280, 16, 50, 3, 1),
    (0, 32, 1, 64, 106_497, 5_000, 200, 300, 170, 8, 20, 2, 1),
    (0, 32, 2, 40, 107_001, 8_000, 90, 120, 25, 16, 64, 0, 1),
    (0, 64, 2, 32, 6_000, 24_000, 1, 70, 256, 1, 5_900, 0, 1),       # fewer candidates than 1.5 n_prune
]
PARAMETERS = "cut,D,nbits,nq,K,N,len_lo,len_hi,B,nprobe,n_prune,shift,copies"


def corpus(D, nbits, nq, K, N, len_lo, len_hi, shift, copies):
    """Arrays on the host and an index of them whose centroid ids start `shift` places behind a 16-byte boundary."""
    import paper_2608_23553_b200 as pkg
    cent, cids, codes, doclens = random_corpus(300 + nq + D, N // copies, K, D, nbits, len_lo=len_lo, len_hi=len_hi)
    if copies > 1:
        cids, codes, doclens = (np.concatenate([a] * copies) for a in (cids, codes, doclens))
    padded = torch.zeros(shift + len(cids), dtype=torch.int32, device="cuda")
    padded[shift:] = torch.from_numpy(cids).cuda()
    gix = pkg.Index(torch.from_numpy(cent).cuda(), padded[shift:], torch.from_numpy(codes).cuda(),
                    torch.from_numpy(doclens).cuda(), nbits)
    return cent, cids, codes, doclens, gix


def queries(cent, B, nq):
    rng = np.random.default_rng(nq)
    K, D = cent.shape
    q = cent[rng.integers(0, K, size=(B, nq))] + 0.3 / np.sqrt(D) * rng.standard_normal((B, nq, D)).astype(np.float32)
    return (q / np.linalg.norm(q, axis=2, keepdims=True)).astype(np.float32)


@pytest.mark.parametrize(PARAMETERS, CALLS)
def test_filtered_searches_match_the_oracle(cut, D, nbits, nq, K, N, len_lo, len_hi, B, nprobe, n_prune, shift, copies):
    cent, cids, codes, doclens, gix = corpus(D, nbits, nq, K, N, len_lo, len_hi, shift, copies)
    oix = oracle.make_index(cent, cids, codes, doclens, nbits)
    q = queries(cent, B, nq)
    k = min(n_prune, 25)
    taps = gix.alloc_taps(B, nq, nprobe, n_prune, table=False)
    ids, sc = gix.search(torch.from_numpy(q).cuda(), nprobe, n_prune, k, taps=taps)
    assert gix.status() == 0
    tn = taps_to_numpy(taps)
    kept = np.array(gix.kept(B, nq, nprobe, n_prune, k))
    assert (kept.sum() < 0.7 * tn["n_cand"].sum() and (kept <= tn["n_cand"]).all()) if cut else (kept == -1).all()
    ids, sc = ids.cpu().numpy(), sc.cpu().numpy()
    for b in (0, B - 1):
        res = oracle.pipeline(q[b], oix, nprobe, n_prune, k)
        check_query(tn, b, res, ids[b], sc[b], k, n_prune, table=False)


@pytest.mark.parametrize(PARAMETERS, [c for c in CALLS if c[0]])
def test_candidates_from_the_caller_are_cut_one_query_at_a_time(cut, D, nbits, nq, K, N, len_lo, len_hi, B, nprobe, n_prune, shift, copies):
    """Stages 3 to 5 on the table and the candidates of a search (whose results the test above checks): the scan by query in all its
    forms, where the search scanned all queries together."""
    cent, _, _, _, gix = corpus(D, nbits, nq, K, N, len_lo, len_hi, shift, copies)
    q = torch.from_numpy(queries(cent, B, nq)).cuda()
    k = min(n_prune, 25)
    taps = gix.alloc_taps(B, nq, nprobe, n_prune, ci=False)
    whole = [t.clone() for t in gix.search(q, nprobe, n_prune, k, taps=taps)]
    pruned, n_pruned, n_cand = taps.pruned.clone(), taps.n_pruned.clone(), taps.n_cand.clone()
    taps.pruned.fill_(-2)
    got = gix.run_stages(3, 5, q, B, nq, nprobe, n_prune, k, taps)
    assert gix.status() == 0
    kept = np.array(gix.kept(B, nq, nprobe, n_prune, k))
    assert kept.sum() < 0.7 * int(n_cand.sum()) and (kept <= n_cand.cpu().numpy()).all()
    assert torch.equal(taps.pruned, pruned) and torch.equal(taps.n_pruned, n_pruned)
    assert torch.equal(got[0], whole[0]) and torch.equal(got[1], whole[1])


@pytest.mark.parametrize("nq", [32, 21])
def test_queries_with_few_candidates_in_a_batch_that_is_cut(nq):
    """The first query has more candidates than n_prune but fewer than the cut wants seeds, the last one fewer than n_prune."""
    import paper_2608_23553_b200 as pkg
    D, K, N, B, n_prune, k = 64, 2_000, 20_000, 260, 300, 20
    cent, cids, codes, doclens = random_corpus(77, N, K, D, 2, len_lo=30, len_hi=50)
    rng = np.random.default_rng(5)
    cids = rng.integers(64, K, size=len(cids)).astype(np.int32)           # centroids 0 ... 63 only where they are put:
    first = np.concatenate([[0], np.cumsum(doclens)[:-1]])
    docs = rng.permutation(N)
    cids[first[docs[:420]]] = rng.integers(0, nq, size=420)
    cids[first[docs[420:520]]] = rng.integers(32, 32 + nq, size=100)
    oix = oracle.make_index(cent, cids, codes, doclens, 2)
    gix = pkg.Index(*(torch.from_numpy(a).cuda() for a in (cent, cids, codes, doclens)), 2)
    c = rng.integers(64, K, size=(B, nq))
    c[0], c[-1] = np.arange(nq), 32 + np.arange(nq)
    q = cent[c].copy()
    taps = gix.alloc_taps(B, nq, 1, n_prune, table=False)
    ids, sc = gix.search(torch.from_numpy(q).cuda(), 1, n_prune, k, taps=taps)
    assert gix.status() == 0
    tn = taps_to_numpy(taps)
    assert sum(gix.kept(B, nq, 1, n_prune, k)) < 0.7 * tn["n_cand"].sum()
    assert n_prune < tn["n_cand"][0] < 1.5 * n_prune and 0 < tn["n_cand"][-1] < n_prune and tn["n_cand"][1] > 1_000
    for b in (0, 1, B - 1):
        res = oracle.pipeline(q[b], oix, 1, n_prune, k)
        check_query(tn, b, res, ids[b].cpu().numpy(), sc[b].cpu().numpy(), k, n_prune, table=False)


# scanned together, q_len, centroids, documents, queries, nprobe
REPEATED = [
    (1, 32, 2_000, 20_000, 260, 2),       # 8-bit rows of a query in shared memory
    (1, 32, 8_000, 20_000, 260, 8),       # ... from L2
    (1, 64, 1_000, 20_000, 100, 1),
    (1, 64, 3_000, 20_000, 200, 2),
    (1, 32, 3_000, 40_000, 31, 8),        # few queries: their contenders over several blocks
    (1, 32, 8_000, 40_000, 37, 16),
    (1, 32, 120_003, 250_000, 100, 60),   # 6-bit codes
    (0, 32, 8_000, 60_000, 260, 3),
    (0, 64, 12_000, 80_000, 130, 2),
]


@pytest.mark.parametrize("together,nq,K,N,B,nprobe", REPEATED)
def test_documents_that_repeat_their_centroids_are_not_cut(together, nq, K, N, B, nprobe):
    """Ten centroids for about forty tokens: nearly all candidates pass the bound, and the call has to notice, whether it would scan all
    queries together or one at a time."""
    import paper_2608_23553_b200 as pkg
    D, n_prune, k = 64, 100, 20
    cent, cids, codes, doclens = random_corpus(K + B, N, K, D, 2, len_lo=30, len_hi=50)
    rng = np.random.default_rng(K)
    own = rng.integers(0, K, size=(N, 10)).astype(np.int32)
    doc = np.repeat(np.arange(N), doclens)
    cids = own[doc, rng.integers(0, 10, size=len(cids))]
    oix = oracle.make_index(cent, cids, codes, doclens, 2)
    gix = pkg.Index(*(torch.from_numpy(a).cuda() for a in (cent, cids, codes, doclens)), 2)
    topic = own[rng.integers(0, N, size=(B, 1)), rng.integers(0, 10, size=(B, nq))]       # half of a query's tokens: one document's
    q = cent[np.where(rng.random((B, nq)) < 0.5, topic, rng.integers(0, K, size=(B, nq)))]
    q = q + 0.3 / np.sqrt(D) * rng.standard_normal(q.shape).astype(np.float32)
    q = (q / np.linalg.norm(q, axis=2, keepdims=True)).astype(np.float32)
    taps = gix.alloc_taps(B, nq, nprobe, n_prune, table=False)
    ids, sc = gix.search(torch.from_numpy(q).cuda(), nprobe, n_prune, k, taps=taps)
    assert gix.status() == 0
    tn = taps_to_numpy(taps)
    assert gix.kept(B, nq, nprobe, n_prune, k) == tn["n_cand"].tolist()
    n_cont = taps.n_contenders.cpu().numpy()
    assert (n_cont < 0.5 * tn["n_cand"]).all()           # the 8-bit bounds narrow them down
    for b in (0, B - 1):
        res = oracle.pipeline(q[b], oix, nprobe, n_prune, k)
        check_query(tn, b, res, ids[b].cpu().numpy(), sc[b].cpu().numpy(), k, n_prune, table=False)
