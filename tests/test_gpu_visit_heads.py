"""Visits kept as lists whose heads hold the last visit: candidates of one visit (known from the head), of several (collected
and walked 32 at a time) and of none, with none, a few and all of them in each share, against the oracle."""
import numpy as np
import pytest
import torch

import oracle
from helpers import random_corpus, unit_rows

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("doclen,repeated", [(1, 0.0), (2, 0.0), (2, 0.1), (2, 1.0), (3, 1.0)])
@pytest.mark.parametrize("N", [2000, 40000])
def test_sums_of_single_and_several_visits(N, doclen, repeated):
    import paper_2608_23553_b200 as pkg
    K, D, nq, nprobe = (1024, 32, 32, 1) if N == 2000 else (4096, 32, 32, 4)
    cent, cids, codes, doclens = random_corpus(N + doclen, N, K, D, 2, len_lo=doclen, len_hi=doclen)
    rng = np.random.default_rng(doclen)
    tok = cids.reshape(N, doclen)
    same = rng.random(N) < repeated
    tok[same] = tok[same][:, :1]                                   # all tokens of these documents share a centroid
    B = torch.cuda.get_device_properties(0).multi_processor_count // 4 + 3
    q = np.stack([unit_rows(rng, nq, D) for _ in range(B)])
    oix = oracle.make_index(cent, cids, codes, doclens, 2)
    gix = pkg.Index(*(torch.from_numpy(a).cuda() for a in (cent, cids, codes, doclens)), 2)
    gix.enable_partial()
    # lists instead of rows of maxima: three more queries take fewer bytes
    assert gix.workspace_bytes(B, nq, nprobe, 50, 5) < gix.workspace_bytes(B - 3, nq, nprobe, 50, 5)
    taps = gix.alloc_taps(B, nq, nprobe, 50, table=False)
    gix.search(torch.from_numpy(q).cuda(), nprobe, 50, 5, taps=taps, partial=True)
    assert gix.status() == 0
    for b in (0, B - 1):
        res = oracle.pipeline(q[b], oix, nprobe, 50, 5, partial=True)
        n = int(taps.n_cand[b])
        assert np.array_equal(taps.cand[b, :n].cpu().numpy(), res.cand)
        assert np.array_equal(taps.ci[b, :n].cpu().numpy(), res.ci.view(np.int32))
