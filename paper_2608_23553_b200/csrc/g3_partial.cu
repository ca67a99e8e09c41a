// Candidate refinement with partial scores (Sec. 3.2 step 2, Algorithm 2; aggregation as in Algorithm 4): only the
// tokens retrieved in candidate generation contribute.  For query token i and each of its probed centroids, every
// token of that centroid's posting list raises M[document, i] to max(M, dist(i, token)); M starts at 0 and the partial
// score is F'(d) = sum_i M[d, i].
//
// dist(i, t) = S[cid_t, i] + llrint(delta*4*T + kappa*4*SQ_i) in Q.24 fixed point, T = sum_x Xq_i[x] u_t[x],
// SQ_i = sum_x Xq_i[x], Xq = rint(q * 2^22): integers plus one correctly rounded double expression, so the result does
// not depend on the order in which tokens are visited (integer max) nor on the machine.
//
// A block serves one query token: one of its posting lists when few queries are served, several or all of them in a batch
// (refine_splits).  The query token's digits sit in shared memory and a thread scores two list entries at a time.  What becomes
// of a score depends on the call:
//   - Batches on large corpora push it onto its candidate's list of visits, which a second kernel sums (g3_visits.cuh).
//   - Few queries per call, small corpora and candidates with many visits keep a table of maxima, one row of q_len per
//     candidate rank (bitmap word prefix + popcount): atomicMax, and every increase is also added to the document's partial
//     score, so that no second kernel is needed.
#include <math.h>

#include "g3_visits.cuh"

namespace chimera {

constexpr int PS_THREADS = 128;

// Nodes per query of the visit lists, 0 when the table of maxima is used: no token lists, few queries per call (latency
// counts), more nodes than their index holds, a table less than three times as large, or candidates with several visits
// each, whose lists are chains of scattered reads: more than two as independent tokens would have them (long documents under
// many probes, where the topics of real ones make it many more), or four by the distinct centroids of a document.
// Whole searches, batch 256 on Mid's sizes, documents that draw 1/4 as many centroids as they have tokens (4.1 visits): lists
// 2.98, table 2.93 ms, 1-bit codes 2.64 / 2.75; an eighth or less (10 visits): 2.96 / 2.68, 2.60 / 2.32; independent (1.1): 3.21 /
// 4.27, 2.83 / 4.71; four topics of near centroids under 32 probes (64 queries): 3.37 / 2.52, 3.05 / 2.45.
// By the ratio of the sizes (batch 256, room for 1.15 times the candidates, residual / 1-bit codes, in us): documents of four topics, 1.9
// lists 2,003 / 1,735, table 1,955 / 1,726; 3.2 2,486 / 2,334 and 2,463 / 2,412; 3.3 (short documents) 1,318 / 1,063 and 1,407 / 1,207;
// independent tokens, where a visit is nearly always a candidate's only one, gain earlier: 1.25 1,796 / 1,450 and 1,816 / 1,450, 2.5 2,419 /
// 2,006 and 2,508 / 2,081, 3.9 1,830 / 1,395 and 2,093 / 1,670.
int64_t visit_list_nodes(const Index &ix, const Params &p)
{
    if (!ix.tok_id || ix.max_tok_list <= 0 || 4 * p.B <= ix.sm_count) return 0;
    const int64_t nodes = (int64_t)p.nq * p.P * ix.max_tok_list;
    if (nodes > VISIT_MAX_NODES) return 0;
    if (3 * 8 * (nodes + p.maxc) > (int64_t)p.maxc * p.nq * 4) return 0;      // (8 bytes a node and a head, 4 an entry of the table)
    const double len = (double)ix.T / (double)ix.N, distinct = (double)ix.ivf_len / (double)ix.N;
    const double probed = (double)p.nq * p.P / (double)ix.K;
    if (len * probed > 1.6) return 0;                    // (visits per candidate: x / (1 - exp(-x)) = 2 at x = 1.6)
    return len * probed <= 4.0 * (1.0 - exp(-distinct * probed)) ? nodes : 0;
}

// Blocks per query token of the refinement kernels: one per probed list until the batch fills the GPU sixteen times over.
int refine_splits(const Index &ix, const Params &p)
{
    int s = (int)((16LL * 8 * ix.sm_count + (int64_t)p.B * p.nq - 1) / ((int64_t)p.B * p.nq));
    return s < 1 ? 1 : s > p.P ? p.P : s;
}

// grid (blocks, B): empty lists for the first n_cand[b] candidates.
__global__ void __launch_bounds__(256)
visit_clear_kernel(unsigned long long *__restrict__ head, const int32_t *__restrict__ n_cand, int64_t maxc)
{
    pdl_entry();
    const int b = blockIdx.y, n = n_cand[b];
    for (int e = blockIdx.x * 256 + threadIdx.x; e < n; e += gridDim.x * 256) head[(int64_t)b * maxc + e] = 0ull;
}
// grid (blocks, B): fprime[b][j] of every candidate.  Walking a list takes some 50 instructions a visit, and nearly every warp
// of 32 candidates has one of several visits: the candidates of one visit or none are written at once, the others collected and
// walked 32 at a time (Mid, batch 256: 226 us with each warp walking its own lists, 134 so).  Long lists
// take turns at the warp's rows of maxima: 8 for up to 32 query tokens, 4 for 64, 2 for 127 (1 KB a warp, which leaves the
// scattered reads their L1; with 2 KB no list gains 1 %).
constexpr int VISIT_ROW_WORDS = 264;                     // 8 x 33, 4 x 65 or 2 x 128
constexpr int VISIT_AHEAD = 4;                           // heads in flight per lane
template <bool FLOAT>
__global__ void __launch_bounds__(256)
visit_sum_kernel(const unsigned long long *__restrict__ head, const unsigned long long *__restrict__ node, int64_t cap,
                 const int32_t *__restrict__ n_cand, int64_t maxc, int nq, int32_t *__restrict__ fprime)
{
    pdl_entry();
    __shared__ uint32_t s_rows[8][VISIT_ROW_WORDS];
    __shared__ unsigned long long s_head[8][64];
    __shared__ int s_place[8][64];
    const int b = blockIdx.y, n = n_cand[b], lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int rows = nq <= 32 ? 8 : nq <= 64 ? 4 : 2, pitch = nq <= 32 ? 33 : nq <= 64 ? 65 : 128;
    const unsigned long long *nodes = node + (int64_t)b * cap;
    const unsigned long long *hb = head + (int64_t)b * maxc;
    int32_t *out = fprime + (int64_t)b * maxc;
    int waiting = 0;                                     // lists collected (uniform)
    auto walk = [&](int m) {                             // the last m of them
        __syncwarp();
        const bool on = lane < m;
        const unsigned long long h = on ? s_head[warp][waiting - m + lane] : 0ull;
        const int place = on ? s_place[warp][waiting - m + lane] : 0;
        waiting -= m;
        int32_t sum;
        const bool done = visit_sum<FLOAT>(h, nodes, sum);
        for (unsigned left = __ballot_sync(0xffffffffu, !done); left;) {
            const int turn = __popc(left & ((1u << lane) - 1));
            const bool mine = (left >> lane & 1u) && turn < rows;
            if (mine) sum = visit_sum_long<FLOAT>(h, nodes, s_rows[warp] + turn * pitch, nq);
            left &= ~__ballot_sync(0xffffffffu, mine);
        }
        if (on) out[place] = sum;
        __syncwarp();
    };
    const int step = gridDim.x * 256;
    for (int j0 = blockIdx.x * 256 + warp * 32; j0 < n; j0 += VISIT_AHEAD * step) {
        unsigned long long h[VISIT_AHEAD];
#pragma unroll
        for (int u = 0; u < VISIT_AHEAD; ++u) h[u] = (int64_t)j0 + u * step + lane < n ? hb[j0 + u * step + lane] : 0ull;
#pragma unroll
        for (int u = 0; u < VISIT_AHEAD; ++u) {
            const int64_t j = (int64_t)j0 + u * step + lane;
            const bool more = (h[u] & VISIT_MORE) != 0;
            if (!more && j < n) out[j] = (int32_t)(h[u] >> 32);
            const unsigned votes = __ballot_sync(0xffffffffu, more);
            if (more) {
                const int at = waiting + __popc(votes & ((1u << lane) - 1));
                s_head[warp][at] = h[u];
                s_place[warp][at] = (int)j;
            }
            waiting += __popc(votes);
            if (waiting >= 32) walk(32);
        }
    }
    if (waiting > 0) walk(waiting);
}
VisitLists visit_lists(const Params &p, const Layout &L, void *mem)
{
    VisitLists v;
    v.cap = L.visit_nodes;
    v.node = (unsigned long long *)mem;
    v.head = v.node + (int64_t)p.B * v.cap;
    return v;
}
int launch_visit_clear(const Index &ix, const Params &p, const VisitLists &v, const int32_t *n_cand, cudaStream_t st)
{
    int64_t gx = (8LL * ix.sm_count + p.B - 1) / p.B;
    launch(visit_clear_kernel, dim3((unsigned)gx, (unsigned)p.B), 256, 0, st, v.head, n_cand, p.maxc);
    CHIMERA_CUDA(cudaGetLastError());
    return CHIMERA_OK;
}
int launch_visit_sum(const Index &ix, const Params &p, const VisitLists &v, bool floats, const int32_t *n_cand,
                     int32_t *fprime, cudaStream_t st)
{
    const dim3 grid((unsigned)((16LL * ix.sm_count + p.B - 1) / p.B), (unsigned)p.B);
    if (floats) launch(visit_sum_kernel<true>, grid, 256, 0, st, v.head, v.node, v.cap, n_cand, p.maxc, p.nq, fprime);
    else launch(visit_sum_kernel<false>, grid, 256, 0, st, v.head, v.node, v.cap, n_cand, p.maxc, p.nq, fprime);
    CHIMERA_CUDA(cudaGetLastError());
    return CHIMERA_OK;
}

// grid (blocks, B): zero the first n_cand[b] rows of M and the first n_cand[b] partial scores.
__global__ void __launch_bounds__(256)
partial_clear_kernel(int32_t *__restrict__ M, int32_t *__restrict__ fprime, const int32_t *__restrict__ n_cand,
                     int64_t maxc, int nq)
{
    pdl_entry();
    const int b = blockIdx.y;
    const int64_t n = (int64_t)n_cand[b] * nq;
    int4 *row = reinterpret_cast<int4 *>(M + (int64_t)b * maxc * nq);      // rows are 16-byte aligned when nq % 4 == 0
    const int64_t tid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, stride = (int64_t)gridDim.x * blockDim.x;
    if ((nq & 3) == 0 && (maxc * nq) % 4 == 0) {
        for (int64_t e = tid; e < n / 4; e += stride) row[e] = make_int4(0, 0, 0, 0);
    } else {
        int32_t *r1 = M + (int64_t)b * maxc * nq;
        for (int64_t e = tid; e < n; e += stride) r1[e] = 0;
    }
    for (int64_t e = tid; e < n_cand[b]; e += stride) fprime[(int64_t)b * maxc + e] = 0;
}

// grid (nq * splits, B): a block takes the lists p, p + splits, ... of a query token (splits = nprobe when few queries are
// served, so that a block is one list; 1 in a large batch, where preparing the query token once per list costs more).
// codes: in list order (tok_id NULL), or the index's document-major codes.
template <int NBITS, bool LISTS>
__global__ void __launch_bounds__(PS_THREADS)
partial_score_kernel(const int8_t *__restrict__ qdig, const int32_t *__restrict__ table, int64_t K, int nq, int B, int CW,
                     int P, float delta, float kappa, const int32_t *__restrict__ probes,
                     const int64_t *__restrict__ tok_off, const int32_t *__restrict__ tok_id,
                     const int32_t *__restrict__ tok_doc, const uint32_t *__restrict__ codes,
                     const uint2 *__restrict__ ranks, int64_t words, int64_t maxc, int32_t *__restrict__ M,
                     int32_t *__restrict__ fprime, VisitLists lists, int64_t longest, int splits)
{
    pdl_entry();
    __shared__ __align__(16) QueryDigits dig;
    const int b = blockIdx.y;
    const int i = blockIdx.x / splits;
    load_query_digits(dig, qdig, table_rows((int64_t)B * nq), table_row((int64_t)b * nq + i));
    __syncthreads();
    const double d4 = __dmul_rn((double)delta, 4.0);
    const double kterm = __dmul_rn(__dmul_rn((double)kappa, 4.0), (double)query_sum(dig));
    const uint2 *rk = ranks + (int64_t)b * words;
    int32_t *Mb = LISTS ? nullptr : M + (int64_t)b * maxc * nq;
    unsigned long long *heads = LISTS ? lists.head + (int64_t)b * maxc : nullptr;
    unsigned long long *nodes = LISTS ? lists.node + (int64_t)b * lists.cap : nullptr;
    int32_t s_c;
    uint32_t v0;                                       // node of the list's first entry
    int64_t e0;
    // (the document's bitmap word and rank come as an argument: they depend on the list entry alone, so their load is
    // issued with the code loads instead of after the score is known -- one memory latency less per visit)
    VisitPush push[2];
    auto update = [&](int n, int64_t e, uint32_t d, int T, uint2 r) {
        const double x = __dadd_rn(__dmul_rn(d4, (double)T), kterm);
        const long long dist = (long long)s_c + __double2ll_rn(x);
        if (dist > 0) {                                // the table starts at 0 (Algorithm 2)
            const int64_t rank = (int64_t)r.y + __popc(r.x & ((1u << (d & 31)) - 1u));
            if (rank < maxc && DBG_RANK_OK(rank)) {
                if (LISTS) {
                    visit_begin(push[n], heads + rank, v0 + (uint32_t)(e - e0), i, (uint32_t)dist);
                } else {
                    // F' = sum_i M[., i] is kept up to date with the increments: M only grows, integer adds commute
                    const int32_t old = atomicMax(&Mb[rank * nq + i], (int32_t)dist);
                    if ((int32_t)dist > old) atomicAdd(&fprime[(int64_t)b * maxc + rank], (int32_t)dist - old);
                }
            }
        }
    };
    for (int p = blockIdx.x % splits; p < P; p += splits) {
        const int32_t c = DBG_CID(probes[((int64_t)b * nq + i) * P + p]);
        s_c = table[((int64_t)b * K + c) * nq + i];
        v0 = (uint32_t)((i * P + p) * longest);
        e0 = tok_off[c];
        const int64_t e1 = tok_off[c + 1];
        // two visits per thread and iteration, their loads issued together (the second one past the end repeats the first)
        for (int64_t e = e0 + threadIdx.x; e < e1; e += 2 * PS_THREADS) {
            const int64_t at[2] = {e, e + PS_THREADS < e1 ? e + PS_THREADS : e};
            uint32_t d[2], w[2][CODE_WORDS<NBITS>];
            uint2 r[2];
#pragma unroll
            for (int n = 0; n < 2; ++n) {
                load_code<NBITS>(w[n], codes + DBG_TOK(tok_id ? (int64_t)tok_id[at[n]] : at[n]) * CW, CW);
                d[n] = (uint32_t)DBG_DOC(tok_doc[at[n]]);
                r[n] = __ldg(rk + (d[n] >> 5));
            }
            if (LISTS) { visit_end(push[0], nodes); visit_end(push[1], nodes); }
            int T[2];
            code_dots<NBITS, 2>(T, w, CW, dig);
            update(0, at[0], d[0], T[0], r[0]);
            if (at[1] != e) update(1, at[1], d[1], T[1], r[1]);
        }
    }
    if (LISTS) { visit_end(push[0], nodes); visit_end(push[1], nodes); }
}

int launch_partial_scores(const Index &ix, const Params &p, const Layout &L, const int8_t *qdig,
                          const int32_t *table, const int32_t *probes, const uint2 *ranks, const int32_t *n_cand,
                          void *partial_m, int32_t *fprime, cudaStream_t st)
{
    const float delta = (ix.res_hi - ix.res_lo) / (float)(1 << ix.nbits);
    const float kappa = ix.res_lo + 0.5f * delta;
    const bool use_lists = L.visit_nodes > 0;
    const VisitLists lists = visit_lists(p, L, partial_m);
    int32_t *M = (int32_t *)partial_m;
    int rc;
    if (use_lists) {
        if ((rc = launch_visit_clear(ix, p, lists, n_cand, st))) return rc;
    } else {
        int64_t per_query = ((int64_t)ix.sm_count * 8 + p.B - 1) / p.B;
        launch(partial_clear_kernel, dim3((unsigned)per_query, (unsigned)p.B), 256, 0, st, M, fprime, n_cand, p.maxc, p.nq);
        CHIMERA_CUDA(cudaGetLastError());
    }
    const int splits = refine_splits(ix, p);
    dim3 grid((unsigned)(p.nq * splits), (unsigned)p.B);
    const uint32_t *codes = reinterpret_cast<const uint32_t *>(ix.list_codes ? ix.list_codes : ix.codes);
    const int32_t *ids = ix.list_codes ? nullptr : ix.tok_id;
#define PS_LAUNCH(NB, LS)                                                                                              \
    launch(partial_score_kernel<NB, LS>, grid, PS_THREADS, 0, st, qdig, table, ix.K, p.nq, p.B, ix.CB / 4, p.P, delta, \
                                                              kappa, probes, ix.tok_off, ids, ix.tok_doc, codes, \
                                                              ranks, L.words, p.maxc, M, fprime, lists, ix.max_tok_list, \
                                                              splits)
    if (ix.nbits == 2) {
        if (use_lists) PS_LAUNCH(2, true); else PS_LAUNCH(2, false);
    } else {
        if (use_lists) PS_LAUNCH(1, true); else PS_LAUNCH(1, false);
    }
#undef PS_LAUNCH
    CHIMERA_CUDA(cudaGetLastError());
    if (use_lists && (rc = launch_visit_sum(ix, p, lists, false, n_cand, fprime, st))) return rc;
    count_launch(SLOT_CI, use_lists ? 3 : 2);
    return CHIMERA_OK;
}

}  // namespace chimera
