"""The joint stages 1 and 2a of a search that keeps no score table (1-bit refinement): the scores that reach the bounds go
straight to the queues, row by row of a chunk.  Row counts that are and are not a multiple of the 32 of a tile (the bounds
are padded), and equal query tokens (all eight rows of a chunk pass for the same centroid); the probes are the oracle's top
nprobe by (score descending, centroid id ascending), bit for bit."""
import numpy as np
import pytest
import torch

import oracle
from helpers import random_corpus, unit_rows

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nq,B,nprobe,same", [(4, 1, 32, False), (4, 3, 32, True), (36, 3, 32, False), (32, 2, 32, True),
                                              (40, 5, 16, True), (52, 2, 32, False)])
def test_probes_without_a_table_match_oracle(nq, B, nprobe, same):
    import paper_2608_23553_b200 as pkg
    from synth import CONFIGS, encode_rabitq_1bit, random_rotation
    K, D = 8192 + 130, 64
    cent, cids, codes, doclens = random_corpus(900 + nq, 200, K, D, 2, len_lo=1, len_hi=30)
    rng = np.random.default_rng(nq + B)
    P = random_rotation(CONFIGS["tiny"].replace(dim=D, seed=3))
    bits, inv = encode_rabitq_1bit(torch.from_numpy(unit_rows(rng, len(cids), D)), P)
    gix = pkg.Index(*[torch.from_numpy(x).cuda() for x in (cent, cids, codes, doclens)], 2)
    gix.attach_rabitq(P.cuda(), bits.cuda(), inv.cuda())
    assert gix.probe_plan(B, nq, nprobe) > 1                       # enough centroids for the joint form
    q = np.stack([np.repeat(unit_rows(rng, 1, D), nq, 0) if same else unit_rows(rng, nq, D) for _ in range(B)])
    taps = gix.alloc_taps(B, nq, nprobe, 16, table=False)
    gix.search(torch.from_numpy(q).cuda(), nprobe, 16, 4, taps=taps, rabitq=True)
    assert gix.status() == 0
    got = taps.probes.cpu().numpy()
    for b in range(B):
        assert np.array_equal(got[b], oracle.probes(oracle.score_table(q[b], cent), nprobe))
