// Visit lists of the candidate refinements (g3_partial.cu, rabitq.cu).
//
// A refinement visits the tokens of the probed lists; a visit (query token i, token t) gives the candidate that owns t a
// score, of which the largest per (candidate, i) counts.  A candidate has about one visit, so a row of q_len maxima per
// candidate is nearly empty: clearing, updating and summing such rows was most of the refinement's traffic (Mid, batch
// 256: 3.4 GB cleared, 3.4 GB read back).  Here every visit is a node of its candidate's list: one exchange of the list's
// head and one 8-byte store; the visits of a candidate are put together afterwards (visit_sum_kernel).  The head holds the last
// visit itself and the place where that visit left the one before, so a list of one node is known from its head alone, without a scattered
// read (the wider heads cost the pushes 587 -> 623 us and their clearing 20 -> 36, Mid's partial scores, batch 256; the sum gains
// more than that, visit_sum_kernel).  Nearly every list has
// one node on documents of independent tokens, several where documents repeat probed centroids or hold neighbours of one:
// lists of up to six are sorted in registers, longer ones walked once over a row of maxima in shared memory (one walk per
// query token before: batch 256, ten visits each, 2.16 ms of refinement, 0.92 so).  The order of a list does not matter: maxima
// per query token, then the sum in increasing query token.
#pragma once
#include "common.cuh"

namespace chimera {

// visit = score bits << 32 | (its own index + 1) << 7 | query token, scores > 0; node[index] holds the visit before it in the
// list (0: none), and a head with VISIT_MORE has one.  The flag is set by whoever finds a visit in the head, after the exchange:
// whichever visit is the head by then, it has a predecessor too.
constexpr int VISIT_I_BITS = 7;                          // q_len <= 127
constexpr int64_t VISIT_MAX_NODES = (1LL << 25) - 1;     // per query
constexpr unsigned long long VISIT_MORE = 1ull << 63;

struct VisitLists {
    unsigned long long *head;      // [B][maxc]: the last visit, 0 = none
    unsigned long long *node;      // [B][cap]
    int64_t cap;                   // q_len * nprobe * longest list
};

int refine_splits(const Index &ix, const Params &p);                        // (g3_partial.cu)
VisitLists visit_lists(const Params &p, const Layout &L, void *mem);
int launch_visit_clear(const Index &ix, const Params &p, const VisitLists &v, const int32_t *n_cand, cudaStream_t st);
int launch_visit_sum(const Index &ix, const Params &p, const VisitLists &v, bool floats, const int32_t *n_cand,
                     int32_t *fprime, cudaStream_t st);

// In two halves: the exchange's answer comes back hundreds of cycles later, so it is put away behind the loads of the next visits.
// (Put away at once, with the branch on it, every visit of a thread
// waited for the one before: 1-bit codes, Mid, batch 256, 503 us, so 488; residual codes 623 either way.)
struct VisitPush {
    unsigned long long *head = nullptr;                  // of the candidate; NULL: nothing pending
    unsigned long long before;
    uint32_t v;
};
__device__ __forceinline__ void visit_begin(VisitPush &push, unsigned long long *head, uint32_t v, int i, uint32_t score)
{
    push.head = head;
    push.v = v;
    push.before = atomicExch(head, (unsigned long long)score << 32 | (v + 1) << VISIT_I_BITS | (uint32_t)i);
}
__device__ __forceinline__ void visit_end(VisitPush &push, unsigned long long *nodes)
{
    if (push.head) {
        nodes[push.v] = push.before & ~VISIT_MORE;
        if (push.before) atomicOr(push.head, VISIT_MORE);
        push.head = nullptr;
    }
}
// The visit before this one, 0 = none.
__device__ __forceinline__ unsigned long long visit_before(unsigned long long visit, const unsigned long long *nodes)
{
    return nodes[((uint32_t)visit >> VISIT_I_BITS) - 1];
}

// ---- products of packed codes with a query token --------------------------------------------------------------------------
// T = sum_x Xq[x] u[x] from the token's three digit planes (balanced base-256 digits, digit_dim() order: a shift and a mask
// give the code values that one word of digits multiplies) with byte dot products: 4.75 instructions per four dimensions
// instead of twelve for value-by-value multiplication.
struct QueryDigits { int32_t plane[3][32]; };            // in shared memory, 16-byte aligned

// rows of a digit plane array [3][n_rows][128]; whole block (128 threads or more), followed by a barrier of the caller's.
__device__ __forceinline__ void load_query_digits(QueryDigits &s, const int8_t *dig, int64_t n_rows, int64_t row)
{
    const int t = threadIdx.x;
    if (t < 96) s.plane[t >> 5][t & 31] = reinterpret_cast<const int32_t *>(dig + ((t >> 5) * n_rows + row) * 128)[t & 31];
}
// sum_x Xq[x] (whole warp, after the barrier).
__device__ __forceinline__ int query_sum(const QueryDigits &s)
{
    const int lane = threadIdx.x & 31, ones = 0x01010101;
    return __reduce_add_sync(0xffffffffu, __dp4a(s.plane[0][lane], ones, 0) + 256 * __dp4a(s.plane[1][lane], ones, 0) +
                                              65536 * __dp4a(s.plane[2][lane], ones, 0));
}
template <int NBITS> constexpr int CODE_WORDS = NBITS == 2 ? 8 : 4;      // 128 dimensions
// A token's CW code words (rows are as aligned as their size allows).
template <int NBITS>
__device__ __forceinline__ void load_code(uint32_t (&w)[CODE_WORDS<NBITS>], const uint32_t *src, int CW)
{
    constexpr int MAX = CODE_WORDS<NBITS>;
    if (NBITS == 2 && CW == 8) {                         // 32-byte codes (32-byte aligned): one load
        asm volatile("ld.global.nc.v8.u32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                     : "=r"(w[0]), "=r"(w[1]), "=r"(w[2]), "=r"(w[3]), "=r"(w[MAX - 4]), "=r"(w[MAX - 3]), "=r"(w[MAX - 2]),
                       "=r"(w[MAX - 1])
                     : "l"(src));
    } else if ((CW & 3) == 0) {
#pragma unroll
        for (int k = 0; k < MAX; k += 4)
            if (k < CW) {
                const uint4 v = __ldg(reinterpret_cast<const uint4 *>(src + k));
                w[k] = v.x; w[k + 1] = v.y; w[k + 2] = v.z; w[k + 3] = v.w;
            }
    } else if ((CW & 1) == 0) {
#pragma unroll
        for (int k = 0; k < MAX; k += 2)
            if (k < CW) {
                const uint2 v = __ldg(reinterpret_cast<const uint2 *>(src + k));
                w[k] = v.x; w[k + 1] = v.y;
            }
    } else {
#pragma unroll
        for (int k = 0; k < MAX; ++k)
            if (k < CW) w[k] = __ldg(src + k);
    }
}
// T of N tokens at once (they share the reads of the digits).  |T| <= 3 * 2^22 * |q|_1 < 2^31 for unit-norm queries.
template <int NBITS, int N>
__device__ __forceinline__ void code_dots(int (&T)[N], const uint32_t (&w)[N][CODE_WORDS<NBITS>], int CW, const QueryDigits &s)
{
    constexpr int PER = 4 * NBITS == 8 ? 4 : 8;          // words of digits per code word
    constexpr uint32_t MASK = NBITS == 2 ? 0x03030303u : 0x01010101u;
    int acc[N][3] = {};
#pragma unroll
    for (int k = 0; k < CODE_WORDS<NBITS>; ++k) {
        if (k < CW) {
#pragma unroll
            for (int h = 0; h < PER; h += 4) {
                int4 d[3];
#pragma unroll
                for (int p = 0; p < 3; ++p) d[p] = *reinterpret_cast<const int4 *>(&s.plane[p][PER * k + h]);
#pragma unroll
                for (int n = 0; n < N; ++n) {
                    const uint32_t word = w[n][k] >> (NBITS * h);
                    const int u[4] = {(int)(word & MASK), (int)(word >> NBITS & MASK), (int)(word >> 2 * NBITS & MASK),
                                      (int)(word >> 3 * NBITS & MASK)};
#pragma unroll
                    for (int p = 0; p < 3; ++p) {
                        acc[n][p] = __dp4a(u[0], d[p].x, acc[n][p]);
                        acc[n][p] = __dp4a(u[1], d[p].y, acc[n][p]);
                        acc[n][p] = __dp4a(u[2], d[p].z, acc[n][p]);
                        acc[n][p] = __dp4a(u[3], d[p].w, acc[n][p]);
                    }
                }
            }
        }
    }
#pragma unroll
    for (int n = 0; n < N; ++n) T[n] = acc[n][0] + 256 * acc[n][1] + 65536 * acc[n][2];
}

// Largest score per query token, summed in increasing query token.  FLOAT: the scores are float bits > 0 (whose order is
// that of the integers) and the sum is a chain of fp32 additions from 0.  Lists of up to six visits; false: a longer one.
template <bool FLOAT>
__device__ __forceinline__ bool visit_sum(unsigned long long head, const unsigned long long *nodes, int32_t &sum)
{
    if (!(head & VISIT_MORE)) {                          // no visit or one; 0.0f + x = x
        sum = (int32_t)(head >> 32);
        return true;
    }
    head &= ~VISIT_MORE;
    constexpr int KEPT = 6;
    // a visit as (query token, score): sorting descending puts the largest score of a query token first
    unsigned long long key[KEPT];
#pragma unroll
    for (int k = 0; k < KEPT; ++k) key[k] = ~0ull;
    auto key_of = [](unsigned long long n) { return (n & ((1ull << VISIT_I_BITS) - 1)) << 32 | (uint32_t)~(uint32_t)(n >> 32); };
    key[0] = key_of(head);
    int cnt = 1;
    unsigned long long n = visit_before(head, nodes);
    while (n != 0 && cnt < KEPT) {
        unsigned long long x = key_of(n);                // ascending (query token, inverted score)
#pragma unroll
        for (int k = 0; k < KEPT; ++k) {
            const unsigned long long lo = x < key[k] ? x : key[k];
            x = x < key[k] ? key[k] : x;
            key[k] = lo;
        }
        ++cnt;
        n = visit_before(n, nodes);
    }
    if (n != 0) return false;
    sum = 0;
    float fs = 0.0f;
    uint32_t last = ~0u;
#pragma unroll
    for (int k = 0; k < KEPT; ++k)
        if (k < cnt && (uint32_t)(key[k] >> 32) != last) {
            last = (uint32_t)(key[k] >> 32);
            const uint32_t score = ~(uint32_t)key[k];
            if (FLOAT) fs = __fadd_rn(fs, __uint_as_float(score));
            else sum += (int32_t)score;
        }
    if (FLOAT) sum = __float_as_int(fs);
    return true;
}

// The same of a list of any length, walked once: row = q_len words of shared memory (a query token without a visit adds 0).
template <bool FLOAT>
__device__ __forceinline__ int32_t visit_sum_long(unsigned long long head, const unsigned long long *nodes, uint32_t *row, int nq)
{
    for (int i = 0; i < nq; ++i) row[i] = 0u;
    for (unsigned long long n = head & ~VISIT_MORE; n != 0; n = visit_before(n, nodes)) {
        const int i = (int)(n & ((1u << VISIT_I_BITS) - 1));
        row[i] = max(row[i], (uint32_t)(n >> 32));
    }
    float fs = 0.0f;
    int32_t is = 0;
    for (int i = 0; i < nq; ++i) {
        if (FLOAT) fs = __fadd_rn(fs, __uint_as_float(row[i]));
        else is += (int32_t)row[i];
    }
    return FLOAT ? __float_as_int(fs) : is;
}

}  // namespace chimera
