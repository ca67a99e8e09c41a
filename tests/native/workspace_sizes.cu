// Workspace of a search for the sizes on standard input, one line each: n_centroids n_docs n_tokens n_queries q_len nprobe n_prune
// max_candidates longest_token_list.  Output: bytes without token lists, with them, of the visit lists or the table of maxima, and
// of the words that lead from a document to its candidate.  Host only.
#include <stdio.h>

#include "common.cuh"

int main()
{
    long long K, N, T, maxc, longest;
    int B, nq, P, n_prune;
    while (scanf("%lld %lld %lld %d %d %d %d %lld %lld", &K, &N, &T, &B, &nq, &P, &n_prune, &maxc, &longest) == 9) {
        chimera::Index ix;
        ix.K = K; ix.N = N; ix.T = T; ix.ivf_len = T; ix.max_doclen = (int32_t)(2 * T / N); ix.sm_count = 148; ix.D = 128; ix.nbits = 2;
        chimera::Params p;
        p.B = B; p.nq = nq; p.P = P; p.n_prune = n_prune; p.k = 10; p.maxc = maxc == 0 || maxc > N ? N : maxc;
        const size_t without = chimera::make_layout(ix, p).total;
        int32_t id;
        ix.tok_id = &id; ix.max_tok_list = longest;
        const chimera::Layout L = chimera::make_layout(ix, p);
        const long long scores = L.visit_nodes ? (L.visit_nodes + p.maxc) * 8 * B : p.maxc * nq * 4 * B;
        printf("%zu %zu %lld %lld\n", without, L.total, scores, (long long)L.words * 8 * B);
    }
    return 0;
}
