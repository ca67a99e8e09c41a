"""The first cut's scan of a whole batch (one pass over the corpus for all queries): every row width, corpora that end inside a
tile or a bitmap word, documents up to the longest that 16-bit sums hold, more listed centroids than there is room for,
and a candidate list that is cut off; candidates, exact scores and selections against the oracle."""
import numpy as np
import pytest

import oracle
from helpers import random_corpus
from parity import check_query, taps_to_numpy

# D, q_len, centroids, documents, shortest, longest, queries, nprobe, n_prune  (80,000 documents: other lengths than 32 and 64 take this
# form from 3 million saved token cycles on, batch_scan_used)
CALLS = [
    (32, 21, 700, 80_000, 1, 99, 8, 8, 100),             # 8-byte rows
    (32, 32, 900, 64 * 400 + 1, 30, 99, 16, 8, 60),      # 16; one document behind the last whole tile
    (64, 64, 1_001, 64 * 300 - 1, 40, 90, 32, 4, 60),    # 32
    (32, 32, 900, 64 * 250 + 33, 1, 120, 61, 8, 50),     # 64
    (32, 100, 1_500, 9_001, 10, 70, 97, 4, 200),         # 128
    (64, 32, 2_000, 12_345, 20, 80, 129, 8, 100),        # 256, half of them empty
    (32, 32, 513, 7_777, 1, 99, 259, 4, 80),             # two groups
    (32, 32, 2_049, 3_000, 900, 1_040, 24, 2, 40),       # the longest documents
    (96, 47, 700, 80_001, 1, 90, 9, 6, 60),
]


def corpus(D, nq, K, N, lo, hi, B, nprobe, n_prune):
    cent, cids, codes, doclens = random_corpus(N + K, N, K, D, 2, len_lo=lo, len_hi=hi)
    return cent, cids, codes, doclens


def tokens_and_entries(*call):
    _, cids, _, doclens = corpus(*call)
    doc = np.repeat(np.arange(len(doclens), dtype=np.int64), doclens)
    return len(cids), len(np.unique(doc * call[2] + cids)), int(doclens.max())


def queries(rng, cent, B, nq):
    D = cent.shape[1]
    q = cent[rng.integers(0, len(cent), size=(B, nq))] + 0.3 / np.sqrt(D) * rng.standard_normal((B, nq, D)).astype(np.float32)
    return (q / np.linalg.norm(q, axis=2, keepdims=True)).astype(np.float32)


def check(arrays, q, nprobe, n_prune, cut=True):
    import torch
    import paper_2608_23553_b200 as pkg
    B, nq, _ = q.shape
    oix = oracle.make_index(*arrays, 2)
    gix = pkg.Index(*(torch.from_numpy(a).cuda() for a in arrays), 2)
    k = min(n_prune, 25)
    taps = gix.alloc_taps(B, nq, nprobe, n_prune, table=False)
    ids, sc = gix.search(torch.from_numpy(q).cuda(), nprobe, n_prune, k, taps=taps)
    assert gix.status() == 0
    tn = taps_to_numpy(taps)
    if cut:
        kept = np.array(gix.kept(B, nq, nprobe, n_prune, k))
        assert kept.sum() < 0.8 * tn["n_cand"].sum() and (kept <= tn["n_cand"]).all()
    ids, sc = ids.cpu().numpy(), sc.cpu().numpy()
    for b in sorted({0, 1, B // 3, B // 2, B - 1}):
        res = oracle.pipeline(q[b], oix, nprobe, n_prune, k)
        check_query(tn, b, res, ids[b], sc[b], k, n_prune, table=False)
    return gix, tn


@pytest.mark.gpu
@pytest.mark.parametrize("call", CALLS)
def test_batches_scanned_together_match_the_oracle(call):
    arrays = corpus(*call)
    check(arrays, queries(np.random.default_rng(call[1]), arrays[0], call[6], call[1]), call[7], call[8])


CROWDED = (32, 8_192, 6_000, 60, 140, 60, 16, 50)        # D, centroids, documents, shortest, longest, queries, nprobe, n_prune


@pytest.mark.gpu
@pytest.mark.parametrize("nq", [20, 32, 64])
def test_more_listed_centroids_than_there_is_room_for(nq):
    """Four thousand centroids near one direction, at odd places, which neither sample looks at (every second centroid for the
    thresholds, every fourth for the step); every query has tokens there, and a fiftieth of the documents' tokens."""
    rng = np.random.default_rng(nq)
    D, K, N, lo, hi, B, nprobe, n_prune = CROWDED
    cent, cids, codes, doclens = random_corpus(9, N, K, D, 2, len_lo=lo, len_hi=hi)
    near = np.arange(K) % 2 == 1
    cent[near] = cent[4] + 0.9 / np.sqrt(D) * rng.standard_normal((int(near.sum()), D)).astype(np.float32)
    cent[near] /= np.linalg.norm(cent[near], axis=1, keepdims=True)
    far = np.flatnonzero(~near)
    cids = np.where(rng.random(len(cids)) < 0.02, cids, rng.choice(far, len(cids))).astype(np.int32)
    q = queries(rng, cent[far], B, nq)
    q[:, :nq // 2] = queries(rng, cent[near], B, nq // 2)
    gix, _ = check((cent, cids, codes, doclens), q, nprobe, n_prune)
    assert gix.cut_plan(B, nq, nprobe, n_prune, 25) == 64
    assert min(gix.listed(B, nq, nprobe, n_prune, 25)) > 1_024


@pytest.mark.gpu
def test_a_candidate_list_that_is_cut_off():
    """Fewer places than candidates: the call reports it, and the bounds of those past the end are not written anywhere."""
    import torch
    import paper_2608_23553_b200 as pkg
    arrays = corpus(*CALLS[3])
    nq, B, nprobe, n_prune = 32, 61, 8, 50
    gix = pkg.Index(*(torch.from_numpy(a).cuda() for a in arrays), 2)
    q = torch.from_numpy(queries(np.random.default_rng(1), arrays[0], B, nq)).cuda()
    whole = gix.alloc_taps(B, nq, nprobe, n_prune, table=False)
    gix.search(q, nprobe, n_prune, 10, taps=whole)
    room = int(whole.n_cand.min()) - 1_000
    cut = gix.alloc_taps(B, nq, nprobe, n_prune, room, table=False)
    ids, _ = gix.search(q, nprobe, n_prune, 10, room, taps=cut)
    assert gix.status() != 0 and (cut.n_cand == room).all()
    for b in (0, B - 1):
        assert torch.equal(cut.cand[b, :room], whole.cand[b, :room])
        best = torch.argsort(whole.ci[b, :room], descending=True, stable=True)[:n_prune]
        assert torch.equal(cut.pruned[b].sort().values, whole.cand[b, :room][best].sort().values)
