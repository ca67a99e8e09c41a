"""Candidates with many visits in a call that keeps visits as lists: documents that repeat a probed centroid, up to the visits
that the sum holds in registers, one more, and hundreds; each size of the rows that long lists are summed in."""
import numpy as np
import pytest
import torch

import oracle
from helpers import random_corpus

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode,nbits,nq", [("partial", 2, 32), ("partial", 1, 51), ("partial", 2, 101), ("rabitq", 2, 32),
                                           ("rabitq", 2, 64)])
def test_candidates_with_many_visits(mode, nbits, nq):
    import paper_2608_23553_b200 as pkg
    from synth import CONFIGS, encode_rabitq_1bit, random_rotation
    D, K, N, nprobe, n_prune, k = 64, 4096, 30_000, 2, 300, 20
    cent, cids, codes, doclens = random_corpus(11 + nbits, N, K, D, nbits, len_lo=20, len_hi=40)
    rng = np.random.default_rng(1)
    first = np.concatenate([[0], np.cumsum(doclens)[:-1]])
    B = torch.cuda.get_device_properties(0).multi_processor_count // 4 + 3
    # document 100 i repeats centroid 10 i once, twice, ... twelve times; document 100 i + 1 holds three centroids only
    for i in range(200):
        t = first[100 * i]
        cids[t:t + 1 + i % 12] = 10 * i
        cids[first[100 * i + 1]:first[100 * i + 2]] = 10 * i + rng.integers(0, 3, size=doclens[100 * i + 1])
    rows = 10 * rng.integers(0, 200, size=(B, 1)) + rng.integers(0, 3, size=(B, nq))
    rows[:, 1::2] = rng.integers(0, K, size=(B, nq // 2))
    q = cent[rows] + 0.3 / np.sqrt(D) * rng.standard_normal((B, nq, D)).astype(np.float32)
    q = (q / np.linalg.norm(q, axis=2, keepdims=True)).astype(np.float32)
    oix = oracle.make_index(cent, cids, codes, doclens, nbits)
    gix = pkg.Index(*(torch.from_numpy(a).cuda() for a in (cent, cids, codes, doclens)), nbits)
    if mode == "partial":
        gix.enable_partial()
    else:
        P = random_rotation(CONFIGS["tiny"].replace(dim=D, seed=3))
        raw = cent[cids] + 0.5 / np.sqrt(D) * rng.standard_normal((len(cids), D)).astype(np.float32)
        raw = (raw / np.linalg.norm(raw, axis=1, keepdims=True)).astype(np.float32)
        bits, inv = encode_rabitq_1bit(torch.from_numpy(raw), P)
        rq = oracle.make_rabitq(P, bits, inv)
        gix.attach_rabitq(P.cuda(), bits.cuda(), inv.cuda())
    # lists instead of rows of maxima: three more queries take fewer bytes
    assert gix.workspace_bytes(B, nq, nprobe, n_prune, k) < gix.workspace_bytes(B - 3, nq, nprobe, n_prune, k)
    taps = gix.alloc_taps(B, nq, nprobe, n_prune, table=False)
    ids, sc = gix.search(torch.from_numpy(q).cuda(), nprobe, n_prune, k, taps=taps, **{mode: True})
    assert gix.status() == 0
    seen = set()
    for b in (0, 1, 17, B - 1):
        res = (oracle.pipeline(q[b], oix, nprobe, n_prune, k, partial=True) if mode == "partial" else
               oracle.pipeline_rabitq(q[b], oix, rq, nprobe, n_prune, k))
        n = int(taps.n_cand[b])
        assert np.array_equal(taps.cand[b, :n].cpu().numpy(), res.cand)
        assert np.array_equal(taps.ci[b, :n].cpu().numpy(), res.ci.view(np.int32))
        assert np.array_equal(taps.pruned[b, :int(taps.n_pruned[b])].cpu().numpy(), res.pruned)
        if mode == "rabitq":
            assert np.array_equal(ids[b].cpu().numpy(), res.ids) and np.array_equal(sc[b].cpu().numpy(), res.scores)
        # visits of each candidate: its tokens in each query token's probed lists
        probed = np.bincount(res.probes.ravel(), minlength=K)
        visits = np.add.reduceat(probed[cids], first)
        seen |= set(visits[res.cand].tolist())
    assert {1, 2, 6, 7} <= seen and max(seen) > 100
