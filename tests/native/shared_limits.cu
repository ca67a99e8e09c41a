// The limits on dynamic shared memory that searches of many sizes set (host only: fake_cudart.cpp).  A limit belongs to the kernel:
// two calls that set unlike ones cannot run on two threads.  Every kernel's limit has to be one number, and enough for its launches.
#include <stdio.h>

#include <map>
#include <set>

#include "common.cuh"

// fake_cudart.cpp
extern std::map<const void *, std::set<int>> fake_limits;
extern std::map<const void *, std::set<size_t>> fake_shared;

using namespace chimera;

int main()
{
    int calls = 0, bad = 0;
    // centroids, documents, tokens of each, queries, q_len, nprobe, n_prune, k
    const long long sizes[][8] = {
        {900, 2'000, 20, 1, 32, 4, 64, 10},          {4'000, 9'000, 100, 16, 32, 32, 300, 100},
        {2'000, 600'000, 90, 16, 64, 32, 500, 200},  {65'536, 500'000, 120, 256, 32, 4, 1'024, 10},
        {65'536, 3'000'000, 120, 256, 64, 48, 1'024, 50}, {262'144, 8'800'000, 68, 256, 32, 64, 4'096, 1'000},
        {120'000, 700'000, 150, 100, 100, 40, 2'000, 500}, {106'000, 900'000, 150, 300, 47, 56, 16'384, 4'000},
        {1'000'000, 400'000, 40, 90, 20, 4, 300, 100},     {16'000, 200'000, 80, 300, 32, 2, 600, 20},
    };
    int32_t word;
    char *ws = nullptr;                                  // (addresses only)
    for (const auto &s : sizes) {
        Index ix;
        ix.K = s[0]; ix.N = s[1]; ix.T = s[1] * s[2]; ix.ivf_len = ix.T; ix.max_doclen = (int32_t)(2 * s[2]);
        ix.D = 128; ix.nbits = 2; ix.CB = 32; ix.sm_count = 148; ix.tok_id = &word; ix.max_tok_list = 2 * ix.T / ix.K;
        ix.graph = &word; ix.graph_deg = 32;
        Params p;
        p.B = (int32_t)s[3]; p.nq = (int32_t)s[4]; p.P = (int32_t)s[5]; p.n_prune = (int32_t)s[6]; p.k = (int32_t)s[7]; p.maxc = s[1];
        const Layout L = make_layout(ix, p);
        const bool batch = batch_scan_used(ix, p);
        const FirstCut cut = first_cut(p, L, ws);
        GraphSearch g;
        g.beam = 64; g.n_entries = 256; g.max_expansions = 100;
        int rc = launch_probes(ix, p, L, nullptr, nullptr, nullptr, nullptr, nullptr);
        if (L.pq_stride) rc |= launch_probe_merge(ix, p, L, nullptr, nullptr, ws, nullptr, nullptr);
        rc |= launch_gather(ix, p, L, nullptr, nullptr, false, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr);
        if (coarse_supported(p.nq)) rc |= launch_coarse_bounds(ix, p, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr);
        if (filter_used(ix, p)) {
            rc |= launch_filter_scan(ix, p, L, batch, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr, ws, nullptr);
            rc |= launch_filter_scan(ix, p, L, false, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr, ws, nullptr);
            rc |= launch_kept_bounds(ix, p, nullptr, filter_mask_used(ix, p, batch) ? (const uint32_t *)&word : nullptr, nullptr, nullptr,
                                     nullptr, nullptr, nullptr, nullptr, nullptr, cut, nullptr);
        }
        for (bool many : {false, true}) rc |= launch_select(ix, p, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr, many, nullptr);
        rc |= launch_topk(ix, p, nullptr, nullptr, nullptr, nullptr, nullptr);
        rc |= launch_graph_probes(ix, nullptr, (int64_t)p.B * p.nq, p.P, g, nullptr, false, nullptr, nullptr, nullptr, nullptr);
        if (rc) { printf("a launch failed\n"); return 2; }
        ++calls;
    }
    int several = 0;
    for (const auto &k : fake_shared) {
        const size_t most = *k.second.rbegin();
        several += most > 48 * 1024 && k.second.size() > 1 ? 1 : 0;
        const auto it = fake_limits.find(k.first);
        if (it == fake_limits.end() ? most > 48 * 1024 : it->second.size() > 1 || (size_t)*it->second.rbegin() < most) {
            printf("a kernel that takes up to %zu bytes:", most);
            if (it != fake_limits.end())
                for (int v : it->second) printf(" %d", v);
            printf(" allowed\n");
            ++bad;
        }
    }
    printf("%d calls, %d kernels that take unlike amounts, %d faults\n", calls, several, bad);
    return bad || several < 6 ? 1 : 0;
}
