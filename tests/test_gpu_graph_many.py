"""Graph search for more query tokens than four-warp blocks are resident (two warps per token then, unless shared memory holds as few
of their blocks), every dimension, short and long lists: probes, scores and visited sets equal the oracle's."""
import numpy as np
import pytest
import torch

import oracle
from helpers import random_corpus, unit_rows

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("K,D,R,B,nq,nprobe,beam,E,max_exp", [
    (2_048, 128, 32, 45, 32, 4, 32, 64, 1 << 30),
    (1_000, 96, 16, 33, 40, 8, 33, 8, 1 << 30),
    (300, 32, 63, 300, 5, 2, 2, 2, 1 << 30),             # all 64 threads of a block have a neighbour, or all but one
    (513, 64, 33, 200, 7, 64, 64, 512, 3),               # more entry points than threads
])
def test_many_tokens(K, D, R, B, nq, nprobe, beam, E, max_exp):
    import paper_2608_23553_b200 as pkg
    cent, cids, codes, doclens = random_corpus(K + nq, 50, K, D, 2)
    gix = pkg.Index(*(torch.from_numpy(a).cuda() for a in (cent, cids, codes, doclens)), 2)
    gix.build_graph(R)
    g = oracle.knn_graph(cent, R)
    rng = np.random.default_rng(K)
    assert B * nq > 8 * torch.cuda.get_device_properties(0).multi_processor_count
    q = cent[rng.integers(0, K, B * nq)] + 0.2 * rng.standard_normal((B * nq, D)).astype(np.float32)
    q[::7] = unit_rows(rng, len(q[::7]), D)
    q = (q / np.linalg.norm(q, axis=1, keepdims=True)).reshape(B, nq, D).astype(np.float32)
    pr, sc, nvis, bm = gix.graph_probes(torch.from_numpy(q).cuda(), nprobe, beam, E, max_exp)
    pr, sc, nvis = pr.cpu().numpy(), sc.cpu().numpy(), nvis.cpu().numpy()
    words = bm.cpu().numpy().view(np.uint32)
    vis = ((words[:, :, None] >> np.arange(32, dtype=np.uint32)) & 1).reshape(B * nq, -1)[:, :K].astype(bool).reshape(B, nq, K)
    for b in range(0, B, max(1, B // 12)):
        o_pr, o_sc, o_vis = oracle.graph_probes(q[b], cent, g, nprobe, beam, E, max_exp)
        assert np.array_equal(pr[b], o_pr) and np.array_equal(sc[b], o_sc)
        assert np.array_equal(vis[b], o_vis) and np.array_equal(nvis[b], o_vis.sum(1))


@pytest.mark.parametrize("beam,E", [(32, 64), (48, 300)])
def test_the_number_of_warps_does_not_change_a_search(beam, E):
    """So many centroids that shared memory bounds the resident blocks: two warps per token for 1,500 tokens, four for 2,100 and for few."""
    import paper_2608_23553_b200 as pkg
    K, D, nq = 140_001, 32, 30
    cent, cids, codes, doclens = random_corpus(3, 50, K, D, 2)
    gix = pkg.Index(*(torch.from_numpy(a).cuda() for a in (cent, cids, codes, doclens)), 2)
    gix.build_graph(32)
    rng = np.random.default_rng(beam)
    q = cent[rng.integers(0, K, 2_100)] + 0.2 * rng.standard_normal((2_100, D)).astype(np.float32)
    q = torch.from_numpy((q / np.linalg.norm(q, axis=1, keepdims=True)).reshape(-1, nq, D).astype(np.float32)).cuda()
    few = [gix.graph_probes(q[b:b + 10].contiguous(), 8, beam, E, 1 << 30) for b in range(0, len(q), 10)]
    few = [torch.cat(x) for x in zip(*few)]
    for b in (50, 70):
        for got, want in zip(gix.graph_probes(q[:b].contiguous(), 8, beam, E, 1 << 30), few):
            assert torch.equal(got, want[:len(got)])
