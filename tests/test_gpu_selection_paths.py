"""Branches that only sizes or ties reach: the top-k that sorts the best entries only, the graph search whose visited set
does not fit shared memory, the RaBitQ search whose score table is made only for the queries that turn out to need it, and
stage 4 for every dimension."""
import numpy as np
import pytest
import torch

import oracle
from helpers import random_corpus, unit_rows

pytestmark = pytest.mark.gpu


def _index(cent, cids, codes, doclens, nbits=2):
    import paper_2608_23553_b200 as pkg
    dev = torch.device("cuda:0")
    return pkg.Index(torch.from_numpy(cent).to(dev), torch.from_numpy(cids).to(dev), torch.from_numpy(codes).to(dev),
                     torch.from_numpy(doclens).to(dev), nbits)


@pytest.mark.parametrize("n,k,distinct", [
    (256, 64, 0), (255, 63, 0), (300, 17, 3), (4096, 100, 0), (4097, 129, 0), (16384, 1000, 0),
    (16384, 4096, 0), (9001, 129, 0), (8192, 2048, 0),
    (16384, 1000, 12),                     # about 1,365 entries per value: the ties fit the second array
    (5000, 513, 5),                        # they do not
])
def test_topk_that_sorts_the_best_entries_only(n, k, distinct):
    gix = _index(*random_corpus(1, 40, 16, 32, 2))
    rng = np.random.default_rng(n + k)
    B, dev = 3, torch.device("cuda:0")
    m = [n, n - 1, k + 1]
    pruned = np.full((B, n), -1, dtype=np.int32)
    score4 = np.full((B, n), -np.inf, dtype=np.float32)
    for b in range(B):
        pruned[b, :m[b]] = rng.permutation(4 * n)[:m[b]]
        score4[b, :m[b]] = rng.integers(0, distinct, m[b]) if distinct else rng.standard_normal(m[b])
    t = gix.alloc_taps(B, 32, 4, n)
    t.pruned, t.n_pruned = torch.from_numpy(pruned).to(dev), torch.tensor(m, dtype=torch.int32, device=dev)
    t.score4 = torch.from_numpy(score4).to(dev)
    ids, sc = gix.run_stages(5, 5, None, B, 32, 4, n, k, t)
    for b in range(B):
        order = np.lexsort((pruned[b, :m[b]], -score4[b, :m[b]].astype(np.float64)))[:k]
        assert np.array_equal(ids[b].cpu().numpy(), pruned[b, order])
        assert np.array_equal(sc[b].cpu().numpy(), score4[b, order])


@pytest.mark.parametrize("K", [1 << 20, (1 << 20) + 1])          # the last count with the bitmap in shared memory, the first without
def test_graph_search_at_the_largest_shared_bitmap(K):
    rng = np.random.default_rng(4)
    cent = unit_rows(rng, K, 32)
    cids = rng.integers(0, K, size=200).astype(np.int32)
    codes = rng.integers(0, 256, size=(200, 8)).astype(np.uint8)
    gix = _index(cent, cids, codes, np.full(20, 10, dtype=np.int32))
    sizes = (2, 8, 4, 10, 5)
    before = gix.workspace_bytes(*sizes)
    gix.build_graph(3)
    vis = 0 if K <= 1 << 20 else 2 * 8 * ((K + 31) // 32) * 4     # a search needs room for the visited sets where they are not shared
    assert vis <= gix.workspace_bytes(*sizes) - before < vis + 256
    q = cent[rng.integers(0, K, size=8)][None] + 0.0
    q[0, -1] = cent[K - 1]
    pr, sc, nvis, bm = gix.graph_probes(torch.from_numpy(q).cuda(), 4, 40, 300, 1 << 30)
    o_pr, o_sc, o_vis = oracle.graph_probes(q[0], cent, gix.graph().cpu().numpy(), 4, 40, 300, 1 << 30)
    assert np.array_equal(pr[0].cpu().numpy(), o_pr) and np.array_equal(sc[0].cpu().numpy(), o_sc)
    words = bm.cpu().numpy().view(np.uint8).reshape(8, -1)
    assert np.array_equal(np.unpackbits(words, axis=1, bitorder="little")[:, :K].astype(bool), o_vis)
    assert np.array_equal(nvis[0].cpu().numpy(), o_vis.sum(1))


def test_rabitq_makes_the_table_for_queries_whose_queue_overflows():
    from synth import CONFIGS, encode_rabitq_1bit, random_rotation
    K, D, nq, nprobe = 33000, 64, 32, 4
    cent, cids, codes, doclens = random_corpus(8, 400, K, D, 2, len_lo=4, len_hi=40)
    cids = (cids % 500).astype(np.int32) * 66
    rng = np.random.default_rng(12)
    hot = unit_rows(rng, 1, D)[0]
    cent[rng.permutation(K)[:30000]] = hot
    P = random_rotation(CONFIGS["tiny"].replace(dim=D, seed=3))
    bits, inv = encode_rabitq_1bit(torch.from_numpy(unit_rows(rng, len(cids), D)), P)
    gix = _index(cent, cids, codes, doclens)
    gix.attach_rabitq(P.cuda(), bits.cuda(), inv.cuda())
    assert gix.probe_plan(3, nq, nprobe) > 1
    q = cent[rng.integers(0, 500, size=(3, nq)) * 66]
    q[0] = unit_rows(rng, nq, D)                                  # far from the copies: its queues suffice
    q[1, :8] = hot
    taps = gix.alloc_taps(3, nq, nprobe, 60, table=False)
    ids, sc = gix.search(torch.from_numpy(q).cuda(), nprobe, 60, 10, taps=taps, rabitq=True)
    assert gix.status() == 0
    oix, rq = oracle.make_index(cent, cids, codes, doclens, 2), oracle.make_rabitq(P, bits, inv)
    for b in range(3):
        assert np.array_equal(taps.probes[b].cpu().numpy(), oracle.probes(oracle.score_table(q[b], cent), nprobe))
        res = oracle.pipeline_rabitq(q[b], oix, rq, nprobe, 60, 10)
        assert np.array_equal(ids[b].cpu().numpy(), res.ids) and np.array_equal(sc[b].cpu().numpy(), res.scores)


@pytest.mark.parametrize("nq", [32, 64])
@pytest.mark.parametrize("D,nbits", [(32, 1), (32, 2), (64, 1), (64, 2), (96, 1), (96, 2), (128, 1)])
def test_stage_4_of_every_dimension(D, nbits, nq):
    """Every document survives, the corpus's last one included, whose code ends with the array."""
    from parity import check_query, taps_to_numpy
    N, nprobe = 97, 16
    cent, cids, codes, doclens = random_corpus(D + nbits, N, 16, D, nbits, len_lo=1, len_hi=150)
    gix = _index(cent, cids, codes, doclens, nbits)
    q = np.stack([unit_rows(np.random.default_rng(7 + b), nq, D) for b in range(2)])
    taps = gix.alloc_taps(2, nq, nprobe, N, table=False)
    ids, sc = gix.search(torch.from_numpy(q).cuda(), nprobe, N, 20, taps=taps)
    assert gix.status() == 0
    oix, tn = oracle.make_index(cent, cids, codes, doclens, nbits), taps_to_numpy(taps)
    for b in range(2):
        check_query(tn, b, oracle.pipeline(q[b], oix, nprobe, N, 20), ids[b].cpu().numpy(), sc[b].cpu().numpy(), 20, N, table=False)
