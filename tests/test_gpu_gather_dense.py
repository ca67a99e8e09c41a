"""Candidates that are a good part of the corpus: bitmaps of more than 48 KB in shared memory, and chunks written word by word."""
import numpy as np
import pytest

from helpers import random_corpus

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,K,B,nprobe,room", [
    (400_003, 64, 2, 16, 0),          # 50 KB, few queries: short chunks
    (400_003, 64, 45, 2, 0),          # chunks of 32,768 documents
    (780_001, 97, 40, 40, 0),         # 95 KB
    (780_001, 97, 40, 5, 50_001),    # ... and a list that ends inside a word
    (50_000, 40, 150, 3, 0),          # a block per query
])
def test_dense_candidates(N, K, B, nprobe, room):
    import torch
    import paper_2608_23553_b200 as pkg
    nq = 32
    cent, cids, codes, doclens = random_corpus(N, N, K, 32, 1, len_lo=1, len_hi=3)
    gix = pkg.Index(*(torch.from_numpy(a).cuda() for a in (cent, cids, codes, doclens)), 1)
    rng = np.random.default_rng(K)
    q = cent[rng.integers(0, K, size=(B, 1))].repeat(nq, axis=1)
    taps = gix.alloc_taps(B, nq, nprobe, 10, room, table=False, ci=False)
    gix.search(torch.from_numpy(np.ascontiguousarray(q)).cuda(), nprobe, 10, 5, room, taps=taps)
    doc = np.repeat(np.arange(N, dtype=np.int32), doclens)
    probes = taps.probes.cpu().numpy()
    for b in (0, B - 1):
        want = np.unique(doc[np.isin(cids, probes[b])])
        n = min(len(want), room) if room else len(want)
        assert int(taps.n_cand[b]) == n
        assert (taps.cand[b, :n].cpu().numpy() == want[:n]).all()
    assert (gix.status() != 0) == bool(room)
