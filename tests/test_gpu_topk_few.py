"""Stage 5 alone for k up to 16: every block size and number of keys per thread, masses of equal scores, padding."""
import numpy as np
import pytest

from helpers import random_corpus

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,k", [(1, 1), (3, 16), (31, 7), (32, 16), (33, 16), (257, 10), (1_023, 1), (1_024, 16), (1_025, 16), (4_096, 10),
                                 (4_097, 3), (16_384, 16)])
@pytest.mark.parametrize("levels", [0, 3])
def test_the_best_few_of_a_list(n, k, levels):
    import torch
    import paper_2608_23553_b200 as pkg
    B, N = 3, 20_000
    cent, cids, codes, doclens = random_corpus(1, N, 50, 32, 1, len_lo=1, len_hi=1)
    gix = pkg.Index(*(torch.from_numpy(a).cuda() for a in (cent, cids, codes, doclens)), 1)
    rng = np.random.default_rng(n + k)
    ids = np.stack([np.sort(rng.choice(N, n, replace=False)) for _ in range(B)]).astype(np.int32)
    sc = rng.standard_normal((B, n)).astype(np.float32)
    if levels:                                           # few distinct scores, both zeros among them
        sc = np.round(sc * levels) / np.float32(levels)
        sc[rng.random((B, n)) < 0.2] = np.float32(-0.0)
    have = rng.integers(0, n + 1, size=B)                # padding behind the survivors
    for b in range(B):
        ids[b, have[b]:], sc[b, have[b]:] = -1, -np.inf
    taps = gix.alloc_taps(B, 32, 1, n, table=False)
    taps.pruned.copy_(torch.from_numpy(ids))
    taps.n_pruned.copy_(torch.from_numpy(have.astype(np.int32)))
    taps.score4.copy_(torch.from_numpy(sc))
    out_ids, out_sc = gix.run_stages(5, 5, None, B, 32, 1, n, k, taps)
    out_ids, out_sc = out_ids.cpu().numpy(), out_sc.cpu().numpy()
    for b in range(B):
        h = int(have[b])
        order = np.lexsort((ids[b, :h], -(sc[b, :h] + 0.0)))[:k]
        want = np.full(k, -1, np.int32)
        want[:len(order)] = ids[b, order]
        assert (out_ids[b] == want).all()
        assert (out_sc[b, :len(order)] == sc[b, order]).all() and np.isneginf(out_sc[b, len(order):]).all()
