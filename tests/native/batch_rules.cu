// Whether the first cut scans a batch at a time (batch_scan_used) for the sizes on standard input, one line each: n_centroids
// n_docs n_tokens posting_entries max_doclen n_queries q_len nprobe n_prune.  Host only.
#include <stdio.h>

#include "common.cuh"

int main()
{
    long long K, N, T, entries, len;
    int B, nq, P, n_prune;
    while (scanf("%lld %lld %lld %lld %lld %d %d %d %d", &K, &N, &T, &entries, &len, &B, &nq, &P, &n_prune) == 9) {
        chimera::Index ix;
        ix.K = K; ix.N = N; ix.T = T; ix.ivf_len = entries; ix.max_doclen = (int32_t)len; ix.sm_count = 148;
        chimera::Params p;
        p.B = B; p.nq = nq; p.P = P; p.n_prune = n_prune; p.k = 1; p.maxc = N;
        printf("%d\n", chimera::batch_scan_used(ix, p) ? 1 : 0);
    }
    return 0;
}
