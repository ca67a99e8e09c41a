"""A corpus of more than 2^31 tokens (no 32-bit token ranges): stages 1 to 3 of a call with few queries."""
import pytest
import torch

pytestmark = pytest.mark.gpu


def test_few_queries_on_more_than_2_31_tokens():
    import paper_2608_23553_b200 as pkg
    from paper_2608_23553_b200 import binding
    if torch.cuda.mem_get_info()[0] < 60 << 30:
        pytest.skip("needs 60 GB of device memory")
    N, length, run, K, D, nq, nprobe, n_prune = 4_400_000, 500, 20, 4096, 32, 32, 2, 700
    T = N * length                                           # runs of equal centroids keep the posting lists short
    g = torch.Generator(device="cuda").manual_seed(3)
    cent = torch.randn(K, D, generator=g, device="cuda")
    cent /= cent.norm(dim=1, keepdim=True)
    cids = torch.randint(0, K, (T // run,), generator=g, device="cuda", dtype=torch.int32).repeat_interleave(run)
    assert cids.numel() == T > 1 << 31
    gix = pkg.Index(cent, cids, torch.zeros(T, D // 8, dtype=torch.uint8, device="cuda"),
                    torch.full((N,), length, dtype=torch.int32, device="cuda"), 1)
    q = cent[torch.randint(0, K, (2, nq), generator=g, device="cuda")].contiguous()
    taps = gix.alloc_taps(2, nq, nprobe, n_prune, table=True)
    binding.profile_read()
    gix.run_stages(1, 3, q, 2, nq, nprobe, n_prune, 10, taps)
    assert gix.status() == 0
    assert binding.profile_read()[1]["select"] == 3 + 1      # the contenders over several blocks per query, the selection
    for b in range(2):
        n = int(taps.n_cand[b])
        assert n > 1_000_000                                 # far more than one block's share
        cand, ci = taps.cand[b, :n].long(), taps.ci[b, :n]
        # centroid interaction of a few documents, the last candidate (token positions past 2^31) among them
        for j in (0, n // 2, n - 1):
            d = int(cand[j])
            rows = taps.score_table[b][cids[d * length:(d + 1) * length].long()]
            assert int(ci[j]) == int(rows.max(dim=0).values.sum())
        order = torch.argsort(ci, descending=True, stable=True)[:n_prune]     # ties: the smaller id, which comes first
        assert torch.equal(taps.pruned[b].long(), cand[order].sort().values)
