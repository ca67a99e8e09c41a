"""Codes in list order: made where there is memory for them, asked for, and searched without."""
import numpy as np
import pytest
import torch

import oracle
from helpers import random_corpus, unit_rows
from parity import check_query, taps_to_numpy

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nbits,batch", [(1, 3), (2, 48)])            # a table of maxima; visit lists
def test_searches_without_the_copies_equal_those_with_them(nbits, batch):
    """The first index is prepared while the device has room for less than four times its copies."""
    import paper_2608_23553_b200 as pkg
    from synth import CONFIGS, encode_rabitq_1bit, random_rotation
    D, nq, K, N, nprobe, n_prune, k = 128, 32, 4096, 24_000, 2, 300, 20
    cent, cids, codes, doclens = random_corpus(90 + nbits, N, K, D, nbits, len_lo=1, len_hi=120)
    oix = oracle.make_index(cent, cids, codes, doclens, nbits)
    rng = np.random.default_rng(3)
    P = random_rotation(CONFIGS["tiny"].replace(dim=D, seed=3))
    bits, inv = encode_rabitq_1bit(torch.from_numpy(unit_rows(rng, len(cids), D)), P)
    arrays = [torch.from_numpy(a).cuda() for a in (cent, cids, codes, doclens)]
    rq = (P.cuda(), bits.cuda(), inv.cuda())
    plain, copied = (pkg.Index(*arrays, nbits) for _ in range(2))
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    smallest = len(cids) * D // 8
    # the lists (8 bytes per token) still fit; allocations come in steps of 2 MB and more
    hog = torch.empty(torch.cuda.mem_get_info()[0] - 3 * smallest - (16 << 20), dtype=torch.uint8, device="cuda")
    assert torch.cuda.mem_get_info()[0] < 4 * smallest
    plain.enable_partial()
    plain.attach_rabitq(*rq)
    assert plain.list_copies() == 0
    del hog
    torch.cuda.empty_cache()
    copied.attach_rabitq(*rq)
    assert copied.list_copies() == 2
    copied.enable_partial()
    assert copied.list_copies() == 3
    q = torch.from_numpy(np.stack([unit_rows(np.random.default_rng(b), nq, D) for b in range(batch)])).cuda()
    for mode in ("partial", "rabitq"):
        out = []
        for ix in (plain, copied):
            taps = ix.alloc_taps(batch, nq, nprobe, n_prune, table=False)
            ids, sc = ix.search(q, nprobe, n_prune, k, taps=taps, **{mode: True})
            assert ix.status() == 0
            out.append((ids, sc, taps))
        assert torch.equal(out[0][0], out[1][0]) and torch.equal(out[0][1], out[1][1])
        for b in (0, batch - 1):
            qb = q[b].cpu().numpy()
            ids, sc = out[0][0][b].cpu().numpy(), out[0][1][b].cpu().numpy()
            if mode == "partial":
                res = oracle.pipeline(qb, oix, nprobe, n_prune, k, partial=True)
                check_query(taps_to_numpy(out[0][2]), b, res, ids, sc, k, n_prune, table=False)
            else:
                res = oracle.pipeline_rabitq(qb, oix, oracle.make_rabitq(P, bits, inv), nprobe, n_prune, k)
                assert np.array_equal(ids, res.ids) and np.array_equal(sc, res.scores)
    # attached again with other codes: the copies are those of the new ones
    bits2, inv2 = encode_rabitq_1bit(torch.from_numpy(unit_rows(rng, len(cids), D)), P)
    copied.attach_rabitq(P.cuda(), bits2.cuda(), inv2.cuda())
    assert copied.list_copies() == 3
    ids, sc = copied.search(q, nprobe, n_prune, k, rabitq=True)
    res = oracle.pipeline_rabitq(q[0].cpu().numpy(), oix, oracle.make_rabitq(P, bits2, inv2), nprobe, n_prune, k)
    assert np.array_equal(ids[0].cpu().numpy(), res.ids) and np.array_equal(sc[0].cpu().numpy(), res.scores)
    # the memory is there now
    plain.enable_partial()
    assert plain.list_copies() == 1
