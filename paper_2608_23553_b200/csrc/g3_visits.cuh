// Visit lists of the candidate refinements (g3_partial.cu, rabitq.cu).
//
// A refinement visits the tokens of the probed lists; a visit (query token i, token t) gives the candidate that owns t a
// score, of which the largest per (candidate, i) counts.  A candidate has about one visit, so a row of q_len maxima per
// candidate is nearly empty: clearing, updating and summing such rows was most of the refinement's traffic (Mid, batch
// 256: 3.4 GB cleared, 3.4 GB read back).  Here every visit is a node of its candidate's list: one exchange of the list's
// head and one 8-byte store; the visits of a candidate are put together afterwards (visit_sum_kernel), where nearly every
// list has one node.  The order of a list does not matter: maxima per query token, then the sum in increasing query token.
#pragma once
#include "common.cuh"

namespace chimera {

// node = score bits << 32 | (index of the next node + 1) << 7 | query token
constexpr int VISIT_I_BITS = 7;                          // q_len <= 127
constexpr int64_t VISIT_MAX_NODES = (1LL << 25) - 1;     // per query

struct VisitLists {
    int32_t *head;                 // [B][maxc]: index of the first node + 1, 0 = empty
    unsigned long long *node;      // [B][cap]
    int64_t cap;                   // q_len * nprobe * longest list
};

int refine_splits(const Index &ix, const Params &p);                        // (g3_partial.cu)
VisitLists visit_lists(const Params &p, const Layout &L, void *mem);
int launch_visit_clear(const Index &ix, const Params &p, const VisitLists &v, const int32_t *n_cand, cudaStream_t st);
int launch_visit_sum(const Index &ix, const Params &p, const VisitLists &v, bool floats, const int32_t *n_cand,
                     int32_t *fprime, cudaStream_t st);

__device__ __forceinline__ void visit_push(int32_t *head /* of the candidate */, unsigned long long *nodes, uint32_t v, int i,
                                           uint32_t score)
{
    const uint32_t next = (uint32_t)atomicExch(head, (int)v + 1);
    nodes[v] = (unsigned long long)score << 32 | next << VISIT_I_BITS | (uint32_t)i;
}

// Largest score per query token, summed in increasing query token.  FLOAT: the scores are float bits > 0 (whose order is
// that of the integers) and the sum is a chain of fp32 additions from 0.
template <bool FLOAT>
__device__ __forceinline__ int32_t visit_sum(int32_t first, const unsigned long long *nodes)
{
    if (first == 0) return 0;                            // (0 is 0.0f as well)
    const unsigned long long n0 = nodes[first - 1];
    uint32_t next = (uint32_t)n0 >> VISIT_I_BITS;
    if (next == 0) return (int32_t)(n0 >> 32);           // one visit; 0.0f + x = x
    float fs = 0.0f;
    int32_t is = 0;
    auto add = [&](uint32_t score) {
        if (FLOAT) fs = __fadd_rn(fs, __uint_as_float(score));
        else is += (int32_t)score;
    };
    constexpr int KEPT = 6;
    // a node as (query token, score): sorting descending puts the largest score of a query token first
    unsigned long long key[KEPT];
#pragma unroll
    for (int k = 0; k < KEPT; ++k) key[k] = ~0ull;
    auto key_of = [](unsigned long long n) { return (n & ((1ull << VISIT_I_BITS) - 1)) << 32 | (uint32_t)~(uint32_t)(n >> 32); };
    key[0] = key_of(n0);
    int cnt = 1;
    while (next != 0 && cnt < KEPT) {
        const unsigned long long n = nodes[next - 1];
        unsigned long long x = key_of(n);                // ascending (query token, inverted score)
#pragma unroll
        for (int k = 0; k < KEPT; ++k) {
            const unsigned long long lo = x < key[k] ? x : key[k];
            x = x < key[k] ? key[k] : x;
            key[k] = lo;
        }
        ++cnt;
        next = (uint32_t)n >> VISIT_I_BITS;
    }
    if (next == 0) {
        uint32_t last = ~0u;
#pragma unroll
        for (int k = 0; k < KEPT; ++k)
            if (k < cnt && (uint32_t)(key[k] >> 32) != last) {
                last = (uint32_t)(key[k] >> 32);
                add(~(uint32_t)key[k]);
            }
    } else {
        // a long list (rare): one walk per query token that occurs in it
        for (int done = -1;;) {
            int at = 1 << VISIT_I_BITS;
            uint32_t best = 0;
            for (uint32_t v = (uint32_t)first; v != 0;) {
                const unsigned long long n = nodes[v - 1];
                const int i = (int)(n & ((1u << VISIT_I_BITS) - 1));
                const uint32_t sc = (uint32_t)(n >> 32);
                if (i > done && (i < at || (i == at && sc > best))) { at = i; best = sc; }
                v = (uint32_t)n >> VISIT_I_BITS;
            }
            if (at == 1 << VISIT_I_BITS) break;
            add(best);
            done = at;
        }
    }
    return FLOAT ? __float_as_int(fs) : is;
}

}  // namespace chimera
