// The routes of stage 3 for the sizes on standard input, one line each: n_centroids n_docs n_tokens posting_entries max_doclen
// n_queries q_len nprobe n_prune max_candidates longest_token_list.  Output: 1 or 0 for the first cut (filter_used), for visit lists
// in the refinements (visit_list_nodes), for bounds from the tokens near the query first (filter_mask_used), for the
// selection of few from many (select_few_used); stage 2b's form (gather_form), and the blocks per query that take all
// rows of the documents that the cut keeps (launch_kept_bounds).  Host only (fake_cudart.cpp).
#include <stdio.h>

#include "common.cuh"

extern unsigned fake_blocks;
void chimera::count_launch(int, int) {}                  // (api.cu's)

int main()
{
    long long K, N, T, entries, len, maxc, longest;
    int B, nq, P, n_prune;
    while (scanf("%lld %lld %lld %lld %lld %d %d %d %d %lld %lld", &K, &N, &T, &entries, &len, &B, &nq, &P, &n_prune, &maxc,
                 &longest) == 11) {
        chimera::Index ix;
        ix.K = K; ix.N = N; ix.T = T; ix.ivf_len = entries; ix.max_doclen = (int32_t)len; ix.sm_count = 148;
        int32_t id;
        ix.tok_id = &id; ix.max_tok_list = longest;
        chimera::Params p;
        p.B = B; p.nq = nq; p.P = P; p.n_prune = n_prune; p.k = 1; p.maxc = maxc == 0 || maxc > N ? N : maxc;
        chimera::launch_kept_bounds(ix, p, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr, chimera::FirstCut(), nullptr);
        printf("%d %d %d %d %d %u\n", chimera::filter_used(ix, p) ? 1 : 0, chimera::visit_list_nodes(ix, p) > 0 ? 1 : 0,
               chimera::filter_mask_used(ix, p, chimera::batch_scan_used(ix, p)) ? 1 : 0, chimera::select_few_used(ix, p) ? 1 : 0,
               chimera::gather_form(ix, p), fake_blocks);
    }
    return 0;
}
