"""Exact scores over token ranges, the next 32 centroid ids always on their way: documents that end around multiples of 32 next to
very short and long ones, as the first, middle and last of a warp's documents, against the oracle."""
import numpy as np
import pytest
import torch

import oracle
from helpers import unit_rows

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lengths", [(32,), (1, 33, 2, 64), (31, 32, 33, 1, 1, 95, 96, 97), (2, 1), (200, 1, 3)])
@pytest.mark.parametrize("nq", [32, 64])
def test_documents_around_multiples_of_32(lengths, nq):
    import paper_2608_23553_b200 as pkg
    from parity import check_query, taps_to_numpy
    N, K, D, nprobe, n_prune, k, B = 3000, 256, 64, 8, 200, 20, 2
    rng = np.random.default_rng(nq + len(lengths))
    dl = np.resize(np.array(lengths, np.int32), N)
    T = int(dl.sum())
    cent = unit_rows(rng, K, D)
    cids = rng.integers(0, K, T).astype(np.int32)
    codes = rng.integers(0, 256, (T, D // 4)).astype(np.uint8)
    gix = pkg.Index(*(torch.from_numpy(a).cuda() for a in (cent, cids, codes, dl)), 2)
    oix = oracle.make_index(cent, cids, codes, dl, 2)
    q = np.stack([unit_rows(rng, nq, D) for _ in range(B)])
    taps = gix.alloc_taps(B, nq, nprobe, n_prune)
    ids, sc = gix.search(torch.from_numpy(q).cuda(), nprobe, n_prune, k, taps=taps)
    assert gix.status() == 0
    tn = taps_to_numpy(taps)
    for b in range(B):
        check_query(tn, b, oracle.pipeline(q[b], oix, nprobe, n_prune, k), ids[b].cpu().numpy(), sc[b].cpu().numpy(), k, n_prune)
