"""The selection of few from many (a sampled bound, one pass, survivors ordered in shared memory) against the rule itself on
the scores that the search reports: the n_prune best by (score descending, id ascending), ids ascending.  Sizes around the
smallest list that takes it, the largest n_prune and beyond; documents that repeat (ties at the edge, more equal scores than
the shared list holds, one score for all)."""
import numpy as np
import pytest
import torch

from helpers import random_corpus, unit_rows

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,n_prune,distinct", [
    (16383, 100, 0), (16384, 100, 0), (16384, 1, 0), (40001, 1024, 0), (40001, 2000, 0), (60000, 4000, 0), (60000, 3000, 0), (60000, 5000, 0),
    (40001, 700, 20000),          # pairs of equal documents, half a pair at the edge now and then
    (40001, 700, 60),             # 667 documents with each score: ties at the edge
    (40001, 700, 5),              # 8,000 with the best score: more than the list holds
    (20000, 300, 1),
    (40001, 700, 8),              # 5,000 with the best score, of which 700 are wanted
    (60000, 4096, 20),            # 3,000 with each score: more ties than the block has threads
    (40001, 3900, 9),             # 4,444 above a bound that as many reach: those above are collected
    (40001, 700, 200),            # 200 with each score: ties counted against one another
])
def test_selected_documents_are_the_best_by_score_then_id(N, n_prune, distinct):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    B, nq = sms // 4 + 1, 8                                        # one block per query
    gix, q = repeating_corpus(N, n_prune, distinct, B, nq)
    taps = gix.alloc_taps(B, nq, 16, n_prune, table=False)         # (all lists of 64: nearly every document is a candidate)
    gix.search(q, 16, n_prune, 1, taps=taps, rabitq=True)
    assert gix.status() == 0
    n_cand, n_pruned = taps.n_cand.cpu().numpy(), taps.n_pruned.cpu().numpy()
    for b in range(B):
        n = int(n_cand[b])
        score, ids = taps.ci[b, :n].cpu().numpy().astype(np.int64), taps.cand[b, :n].cpu().numpy()
        best = np.sort(np.argsort(-score, kind="stable")[:n_prune])
        assert int(n_pruned[b]) == len(best)
        assert np.array_equal(taps.pruned[b, :len(best)].cpu().numpy(), ids[best])
        if distinct != 1:
            assert n > 16000                                       # the sizes above are about this


def test_masses_of_equal_scores_take_no_longer_than_a_few_times_others():
    """2,000 documents with each score and 4,096 wanted, against one of each (one by one and against one another: 11 times as long)."""
    from paper_2608_23553_b200.binding import profile_enable, profile_read
    ms = {}
    for distinct in (0, 20):
        gix, q = repeating_corpus(40000, 4096, distinct, 256, 8)
        gix.search(q, 16, 4096, 1, rabitq=True)
        profile_enable(True)
        profile_read()
        for _ in range(5):
            gix.search(q, 16, 4096, 1, rabitq=True)
        ms[distinct] = profile_read()[0]["select"]
        profile_enable(False)
    assert ms[20] < 3 * ms[0]


def repeating_corpus(N, n_prune, distinct, B, nq):
    """N documents, `distinct` unlike ones (0: all), and B queries."""
    import paper_2608_23553_b200 as pkg
    from synth import CONFIGS, encode_rabitq_1bit, random_rotation
    K, D, L = 64, 32, 4
    rng = np.random.default_rng(N + n_prune + distinct)
    base = distinct if distinct else N
    pick = np.arange(N) % base
    cent, cids, codes, _ = random_corpus(5, base, K, D, 2, len_lo=L, len_hi=L)
    P = random_rotation(CONFIGS["tiny"].replace(dim=D, seed=3))
    bits, inv = encode_rabitq_1bit(torch.from_numpy(unit_rows(rng, base * L, D)), P)
    tok = torch.from_numpy((pick[:, None] * L + np.arange(L)[None, :]).reshape(-1))
    dl = torch.full((N,), L, dtype=torch.int32)
    gix = pkg.Index(torch.from_numpy(cent).cuda(), torch.from_numpy(cids)[tok].cuda(), torch.from_numpy(codes)[tok].cuda(), dl.cuda(), 2)
    gix.attach_rabitq(P.cuda(), bits[tok].contiguous().cuda(), inv[tok].contiguous().cuda())
    return gix, torch.from_numpy(np.stack([unit_rows(rng, nq, D) for _ in range(B)])).cuda()
