// Warps per token of the graph search (graph_search_warps) for the sizes on standard input, one line each: n_centroids n_tokens.
// Host only.
#include <stdio.h>

#include "common.cuh"

int main()
{
    long long K, tokens;
    while (scanf("%lld %lld", &K, &tokens) == 2) {
        chimera::Index ix;
        ix.K = K; ix.sm_count = 148;
        printf("%d\n", chimera::graph_search_warps(ix, tokens));
    }
    return 0;
}
