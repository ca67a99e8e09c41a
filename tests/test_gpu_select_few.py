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
])
def test_selected_documents_are_the_best_by_score_then_id(N, n_prune, distinct):
    import paper_2608_23553_b200 as pkg
    from synth import CONFIGS, encode_rabitq_1bit, random_rotation
    K, D, nq, L = 64, 32, 8, 4
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    B = sms // 4 + 1                                               # one block per query
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
    q = torch.from_numpy(np.stack([unit_rows(rng, nq, D) for _ in range(B)])).cuda()
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
