// Stage 4 on the tensor cores: residual-decode MaxSim of the surviving documents (Definition 1 on the
// decoded tokens),
//   score(d) = sum_i max_{t in d} <q_i, c_{cid_t} + r^(code_t)>
//            = sum_i [ max_t ( S[cid_t, i] + delta * sum_x q_i[x] u_t[x] ) + (lo + delta/2) * sum_x q_i[x] ].
// The code contraction sum_x q_i[x] u_t[x] is a dense [tokens x D] x [D x q_len] product with tiny integer entries on
// one side, so it runs as an exact integer MMA: the bucket indices u (0..3) are int8, the query is the same three
// int8 digit planes of rint(q * 2^22) that stage 1 built, and tcgen05.mma kind::i8 gives sum_x u digit_a exactly in
// int32; the three planes are recombined in fp32 (relative error 2^-24).
//
// A CTA owns one query and a run of its surviving documents, whose tokens form one stream cut into tiles of 128
// (MMA M).  The kernel is bound by the instructions and latencies around the MMAs (tensor pipe 15 %), so:
//   - codes expand with one shift and one mask per four dimensions (the query's digits are stored in the order in which
//     codes expand, digit_dim()) and go into tensor memory as the A operand with one tcgen05.st per thread;
//   - each warp takes 16 query tokens of a quarter's 32 token rows (two warps per quarter for q_len <= 32, four above) and
//     reads the accumulators back in the 16x256b shape, i.e. already spread over (row, four query tokens): the maxima are
//     folded in registers, without a transposition through shared memory, and the score-table entries of the centroid
//     term come as one 16-byte load per row, four lanes to a row (a thread per row would touch 32 lines with each load);
//   - the accumulators of tile t are read back before the tile's only block barrier, and behind it tile t + 1's MMAs, code
//     and row loads run while tile t is folded.
// Measured (batch 256, Mid, n_prune 1024): 2.24 -> 1.56 ms against one warp per quarter, value rows in shared memory and
// two barriers per tile; 64 long-document queries of 64 tokens: 5.9 -> 3.75 ms.  Residency: q_len <= 32 three CTAs of 256
// threads (85 registers, no spills; four with 64 registers: 1.78 ms; the RaBitQ variant, which holds no score-table
// entries, four: 1.18 against 1.32 ms), q_len <= 64 two of 512 threads.  Longer queries
// take two launches (8 queries of 100 tokens, n_prune 1024: 1.91 ms with an FMA kernel, 0.26 with these).  All mbarrier waits are
// bounded.
#include <math.h>

#include "common.cuh"
#include "umma.cuh"

namespace chimera {

constexpr int G4U_COLS = 16;              // query tokens per draining warp
constexpr int G4U_TOK = 128;             // tokens per tile (MMA M)
constexpr int G4U_MAX_DOCS = 32;         // documents per CTA, at most

__device__ __forceinline__ uint32_t f_order(float f)
{
    uint32_t u = __float_as_uint(f);
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
__device__ __forceinline__ float f_unorder(uint32_t o)
{
    return __uint_as_float((o & 0x80000000u) ? (o & 0x7fffffffu) : ~o);
}

// RQ = true scores RaBitQ 1-bit codes instead (Sec. 2.2; the GPU half of the paper's document scoring): the same
// contraction T = sum_x Xq[x] b[x] against the digit planes of the ROTATED query, then
// est = inv_dot_t * (c * (float)(2 T - SQ_i)) with SQ_i = sum_x Xq_i[x] and c = 1 / (sqrt(D) 2^22); no centroid term;
// query tokens are summed in increasing order in fp32 so that the score is reproducible bit for bit.
// DIM: the dimension, so that a code's extent is known when this is compiled (64 queries of 64 tokens, long documents: dim 96
// took 4.36 ms without, 3.96 with it; 64 queries of 32 tokens, Mid with dim 96: 0.60, now 0.41).  FULL: q_len is NQP, no row is
// partial.
template <int NQP, int NBITS, bool RQ, int DIM, bool FULL>
__global__ void __launch_bounds__(128 * (NQP / G4U_COLS), NQP == 32 ? (RQ ? 4 : 3) : 2)
residual_maxsim_umma(const __grid_constant__ CUtensorMap map_q, const float *__restrict__ queries,
                     const int32_t *__restrict__ table, int64_t K, int nq_arg, int q_base, int nq_all_arg, int q_rows, float delta, float kappa,
                     const int32_t *__restrict__ pruned, int n_prune, int docs_per_cta,
                     const int32_t *__restrict__ cids, const uint32_t *__restrict__ codes,
                     const float *__restrict__ factors, const int64_t *__restrict__ doc_off,
                     float *__restrict__ score4, uint32_t *status, long long wait_limit, int skip_loads)
{
    pdl_entry();
    // this launch's query tokens are q_base ... q_base + nq - 1 of the query's nq_all (its digit planes have q_rows rows)
    const int nq = FULL ? NQP : nq_arg, nq_all = FULL ? NQP : nq_all_arg;
    constexpr int D = DIM, CW = DIM * NBITS / 32;
    constexpr int N = 3 * NQP;                               // MMA N: three digit planes side by side
    constexpr uint32_t TMEM_COLS = N <= 96 ? 128 : 256;
    constexpr uint32_t A_COL = N;                            // the expanded codes: 32 columns behind the accumulators
    static_assert(N + 32 <= TMEM_COLS, "accumulators and the A operand share the allocation");
    constexpr uint32_t B_BYTES = N * 128;
    constexpr int WPQ = NQP / G4U_COLS;                      // warps per lane quarter: each drains 16 query tokens
    constexpr int G4U_THREADS = 128 * WPQ;
    constexpr uint32_t IDESC = (2u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) |
                               ((uint32_t)(G4U_TOK >> 4) << 24);

    extern __shared__ uint8_t smem_raw[];
    __shared__ uint32_t s_tmem_base;
    __shared__ int s_abort;
    __shared__ int s_off[G4U_MAX_DOCS + 1];                  // stream offset of each document
    __shared__ long long s_t0[G4U_MAX_DOCS];                 // first global token of each document
    __shared__ float s_sumq[NQP];
    __shared__ int s_sq[NQP];                                // RQ: sum_x rint(q_p[x] * 2^22) per query token
    const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    uint8_t *gen = smem_raw + (base - smem_u32(smem_raw));   // generic pointer to the aligned area
    const uint32_t sB = base;                                                      // [3][NQP][128] int8
    uint32_t *docmax = reinterpret_cast<uint32_t *>(gen + B_BYTES);                // [MAX_DOCS][NQP]
    const uint32_t bars = smem_u32(docmax + G4U_MAX_DOCS * NQP);
    const uint32_t bar_b = (bars + 7u) & ~7u, bar_mma = bar_b + 8;

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int quarter = warp & 3, part = warp >> 2;          // lanes of tensor memory, columns / code words of this warp
    const int row = tid & 127;                               // this thread's token of a tile (shared by the WPQ parts)
    const int b = blockIdx.y;
    const int j0 = blockIdx.x * docs_per_cta;
    int nd = n_prune - j0;
    if (nd > docs_per_cta) nd = docs_per_cta;

    if (tid == 0) {
        mbar_init(bar_b, 1);
        mbar_init(bar_mma, 1);
        s_abort = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        // stream offsets of this CTA's documents (padding slots have id -1 and no tokens): lane = document, one
        // round of loads, then a prefix sum of the lengths
        int32_t d = -1;
        if (lane < nd) d = pruned[(int64_t)b * n_prune + j0 + lane];
        long long t0 = 0;
        int len = 0;
        if (d >= 0) {
            d = DBG_DOC(d);
            t0 = doc_off[d];
            len = (int)(doc_off[d + 1] - t0);
        }
        int incl = len;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int t = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += t;
        }
        if (lane < nd) {
            s_off[lane] = incl - len;
            s_t0[lane] = t0;
        }
        if (lane == 31) s_off[nd] = incl;          // lanes past nd add nothing
    }
    if (warp == 0) {
        __syncwarp();
        tmem_alloc(&s_tmem_base, TMEM_COLS);
    }
    for (int e = tid; e < G4U_MAX_DOCS * NQP; e += G4U_THREADS) docmax[e] = 0u;     // below every real value
    // sum_x q_i[x] per query token: four threads per row, each a quarter of the row with 16-byte loads
    for (int i = tid >> 2; i < NQP; i += G4U_THREADS / 4) {
        float sum = 0.f;
        int si = 0;
        if (i < nq) {
            const int fourth = D >> 2;                // D is a multiple of 32
            const float4 *src = reinterpret_cast<const float4 *>(queries + ((int64_t)b * nq_all + q_base + i) * D + (tid & 3) * fourth);
            for (int x = 0; x < (fourth >> 2); ++x) {
                const float4 v = __ldg(src + x);
                sum += (v.x + v.y) + (v.z + v.w);
                si += __float2int_rn(fminf(fmaxf(v.x, -1.0f), 1.0f) * 4194304.0f) +
                      __float2int_rn(fminf(fmaxf(v.y, -1.0f), 1.0f) * 4194304.0f) +
                      __float2int_rn(fminf(fmaxf(v.z, -1.0f), 1.0f) * 4194304.0f) +
                      __float2int_rn(fminf(fmaxf(v.w, -1.0f), 1.0f) * 4194304.0f);
            }
        }
        sum += __shfl_xor_sync(0xffffffffu, sum, 1);
        si += __shfl_xor_sync(0xffffffffu, si, 1);
        sum += __shfl_xor_sync(0xffffffffu, sum, 2);
        si += __shfl_xor_sync(0xffffffffu, si, 2);
        if ((tid & 3) == 0) { s_sumq[i] = sum; s_sq[i] = si; }
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = s_tmem_base;
    const int total = s_off[nd];
    const int n_tiles = (total + G4U_TOK - 1) / G4U_TOK;

    // skip_loads (test hook): no load is issued, so the first wait below runs into its limit with nothing in flight
    if (tid == 0 && !skip_loads) {   // the query's three digit planes, side by side: rows [p * NQP, (p + 1) * NQP)
        mbar_expect_tx(bar_b, B_BYTES);
        for (int p = 0; p < 3; ++p) tma_load_3d(sB + p * NQP * 128, &map_q, 0, b * q_rows + q_base, p, bar_b);
    }

    const char *tb = reinterpret_cast<const char *>(table + (int64_t)b * K * nq_all + q_base);
    const uint32_t row_bytes = 4u * (uint32_t)nq_all;
    const bool vec_rows = (nq_all & 3) == 0;       // 16-byte groups of a row are aligned (q_base is a multiple of 64)
    const int k_steps = D >> 5;
    const float code_scale = delta * 4.0f;                    // delta * 2^-22, times 2^24
    bool alive = true;
    // Code words of a token that one thread expands: a token has at most 32 code bytes (2 bits per dimension) or 16 (1 bit).
    constexpr int TW = (NBITS == 2 ? 8 : 4) / WPQ;
    constexpr int ACOLS = 32 / WPQ;                           // columns of the A operand they fill
    const int w0 = part * TW;

    // Token of stream position s (this thread's row of a tile): centroid id (-1 past the stream's end) and its part of the
    // packed code.  Positions only move forward, so the document is found by stepping on.
    int at_doc = -1, at_end = 0;
    const uint32_t *at_code = nullptr;                        // of position 0, were it in the same document
    const int32_t *at_cid = nullptr;                          // (RQ: the token's factor, whose bits > 0 take the id's place)
    auto fetch = [&](int tile, int32_t &cid, uint32_t (&cw)[TW]) {
        const int s = tile * G4U_TOK + row;
        cid = -1;
        if (s >= total) return;
        if (s >= at_end) {
            do ++at_doc; while (s_off[at_doc + 1] <= s);
            at_end = s_off[at_doc + 1];
            const long long t = s_t0[at_doc] - s_off[at_doc];
            at_code = codes + t * CW + w0;
            at_cid = (RQ ? reinterpret_cast<const int32_t *>(factors) : cids) + t;
        }
#ifdef CHIMERA_DEBUG
        const long long dbg_t = s_t0[at_doc] + s - s_off[at_doc];
        if (DBG_TOK(dbg_t) != dbg_t) return;                  // (reported; the row keeps no token)
#endif
        cid = __ldg(at_cid + s);
        const uint32_t *src = at_code + (long long)s * CW;
        if (w0 >= CW) {                                       // (this warp's part lies behind a short code)
        } else if (TW == 4 && (CW & 3) == 0) {
            const uint4 v = __ldg(reinterpret_cast<const uint4 *>(src));
            cw[0] = v.x; cw[1] = v.y; cw[TW > 2 ? 2 : 0] = v.z; cw[TW > 3 ? 3 : 0] = v.w;
        } else if (TW >= 2 && (CW & 1) == 0) {
#pragma unroll
            for (int w = 0; w < TW; w += 2)
                if (w0 + w < CW) {
                    const uint2 v = __ldg(reinterpret_cast<const uint2 *>(src + w));
                    cw[w] = v.x; cw[w + 1 < TW ? w + 1 : w] = v.y;
                }
        } else {
#pragma unroll
            for (int w = 0; w < TW; ++w)
                if (w0 + w < CW) cw[w] = __ldg(src + w);
        }
    };

    // Expands this thread's part of a token into lane `row` of the A operand in tensor memory.  A row without a token keeps
    // whatever cw holds (its products take part in no maximum); columns past the code are not multiplied.
    auto expand = [&](const uint32_t (&cw)[TW]) {
        uint32_t a[ACOLS];
#pragma unroll
        for (int w = 0; w < TW; ++w) {
            const uint32_t word = cw[w];
            if (NBITS == 2) {
#pragma unroll
                for (int h = 0; h < 4; ++h) a[4 * w + h] = (word >> (2 * h)) & 0x03030303u;
            } else {
#pragma unroll
                for (int h = 0; h < 8; ++h) a[8 * w + h] = (word >> h) & 0x01010101u;
            }
        }
        tmem_st(tmem + ((uint32_t)(quarter * 32) << 16) + A_COL + part * ACOLS, a);
        asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
    };
    auto issue = [&]() {                                      // one thread
        tc_fence_after();
        const uint64_t db = umma_desc(sB);
        for (int k = 0; k < k_steps; ++k) umma_i8_ts(tmem, tmem + A_COL + 8 * k, db + 2 * k, IDESC, k > 0 ? 1u : 0u);
        umma_commit(bar_mma);
    };

    int fold_doc = -1, fold_end = 0;                          // document of the warp's first token in the tile being folded
    int32_t cid = -1, cid_next = -1;
    uint32_t cw[TW] = {};
    const int grp = lane & 3, sub = lane >> 2;                // fold: four query tokens, a row of every eight
    const int col0 = part * G4U_COLS + 4 * grp;
    // The MMAs of tile t + 1 run while tile t is folded: accumulators are read back and the A operand is rewritten as soon
    // as tile t's MMAs are done, in front of the tile's only block barrier.
    if (n_tiles > 0) {
        fetch(0, cid, cw);
        expand(cw);
        if (n_tiles > 1) fetch(1, cid_next, cw);
        tc_fence_before();
        __syncthreads();
        if (tid == 0) {
            if (mbar_wait(bar_b, 0, wait_limit)) issue();
            else s_abort = 1;
        }
        __syncwarp();
    }

    // Score-table entries of a tile's tokens, in the layout in which the accumulators come back: rows sub, sub + 8, ... of the
    // warp's 32 tokens, query tokens col0 ... col0 + 3.  Four lanes read 64 bytes of a row, so a load of the warp touches
    // eight lines; one thread per row would touch 32 with each.
    int32_t sv[4][4];
    auto load_rows = [&](int32_t cid) {
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            int32_t c = __shfl_sync(0xffffffffu, cid, sub + 8 * j);
            c = DBG_CID(c > 0 ? c : 0);                       // (rows without a token take part in no maximum)
            const int32_t *src = reinterpret_cast<const int32_t *>(tb + (uint64_t)(uint32_t)c * row_bytes) + col0;
            if (FULL || (vec_rows && col0 + 3 < nq)) {
                const int4 q = __ldg(reinterpret_cast<const int4 *>(src));
                sv[j][0] = q.x; sv[j][1] = q.y; sv[j][2] = q.z; sv[j][3] = q.w;
            } else {
#pragma unroll
                for (int e = 0; e < 4; ++e) sv[j][e] = col0 + e < nq ? __ldg(src + e) : 0;
            }
        }
    };
    if (!RQ) load_rows(cid);

    for (int tile = 0; tile < n_tiles; ++tile) {
        // the next token's scattered score-table row misses L2 (a batch's tables are far larger): ask for it now
        // (measured: a gain for q_len <= 32, a loss for the two-line rows of longer queries)
        if (!RQ && NQP == 32 && part == 0 && cid_next >= 0) {
            const char *next = tb + (uint64_t)(uint32_t)DBG_CID(cid_next) * row_bytes;
            for (int off = 0; off < nq * 4; off += 128) asm volatile("prefetch.global.L2 [%0];" ::"l"(next + off));
        }

        const bool ok = mbar_wait(bar_mma, tile & 1, wait_limit);
        tc_fence_after();
        __syncwarp();

        // ---- accumulators -> code products of rows sub + 8 j, query tokens col0 ... col0 + 3 --------------------------------
        const uint32_t lane_addr = tmem + ((uint32_t)(quarter * 32) << 16) + part * G4U_COLS;
        int32_t T[4][4];
#pragma unroll
        for (int half = 0; half < 2; ++half) {
            int32_t a0[8], a1[8], a2[8];
            tmem_ld_16x16(lane_addr + (uint32_t)(half * 16 << 16) + 0 * NQP, a0);
            tmem_ld_16x16(lane_addr + (uint32_t)(half * 16 << 16) + 1 * NQP, a1);
            tmem_ld_16x16(lane_addr + (uint32_t)(half * 16 << 16) + 2 * NQP, a2);
            tmem_ld_wait();
#pragma unroll
            for (int o = 0; o < 8; ++o)
                // |sum_x u_x Xq_x| <= 3 * 2^22 * |q|_1 < 2^31: the plane recombination fits int32
                T[2 * half + (o >> 1 & 1)][(o & 1) + (o >> 2) * 2] = (a2[o] * 256 + a1[o]) * 256 + a0[o];
        }

        // ---- the next tile's codes, its MMAs, the token after it ----------------------------------------------------------
        if (tile + 1 < n_tiles) expand(cw);
        tc_fence_before();
        if (!__syncthreads_and(ok && !*(volatile int *)&s_abort)) {
            if (tid == 0) atomicOr(status, ST_TIMEOUT);
            alive = false;
            break;
        }
        if (tid == 0 && tile + 1 < n_tiles) issue();
        __syncwarp();
        int32_t cid_far = -1;
        if (tile + 2 < n_tiles) fetch(tile + 2, cid_far, cw);

        // ---- values (times 2^24: S is an integer there, and a power of two changes no rounding); the next tile's rows --------
        float v[4][4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const float f = RQ ? __int_as_float(__shfl_sync(0xffffffffu, cid, sub + 8 * j)) : 0.f;
#pragma unroll
            for (int e = 0; e < 4; ++e)
                v[j][e] = RQ ? __fmul_rn(f, __fmul_rn(kappa, (float)(2 * T[j][e] - s_sq[col0 + e])))
                             : fmaf(code_scale, (float)T[j][e], (float)sv[j][e]);
        }
        if (!RQ) load_rows(cid_next);

        // ---- fold the warp's 32 tokens into the per-document maxima ---------------------------------------------------------
        // maximum over the eight lanes of a column group: each exchange keeps half of the columns, the last one is whole
        auto publish = [&](int doc, float m0, float m1, float m2, float m3) {
            const bool up = (lane & 16) != 0, up2 = (lane & 8) != 0;
            const float h0 = fmaxf(up ? m2 : m0, __shfl_xor_sync(0xffffffffu, up ? m0 : m2, 16));
            const float h1 = fmaxf(up ? m3 : m1, __shfl_xor_sync(0xffffffffu, up ? m1 : m3, 16));
            float x = fmaxf(up2 ? h1 : h0, __shfl_xor_sync(0xffffffffu, up2 ? h0 : h1, 8));
            x = fmaxf(x, __shfl_xor_sync(0xffffffffu, x, 4));
            if ((lane & 4) == 0) atomicMax(&docmax[doc * NQP + col0 + (up ? 2 : 0) + (up2 ? 1 : 0)], f_order(x));
        };
        const int s0 = tile * G4U_TOK + quarter * 32;          // first token of the warp
        if (s0 < total) {
            if (s0 >= fold_end) {
                do fold_end = s_off[++fold_doc + 1]; while (fold_end <= s0);
            }
            if (fold_end >= s0 + 32) {
                // all 32 tokens are of one document (most of a long document's)
                float m[4];
#pragma unroll
                for (int e = 0; e < 4; ++e) m[e] = fmaxf(fmaxf(v[0][e], v[1][e]), fmaxf(v[2][e], v[3][e]));
                publish(fold_doc, m[0], m[1], m[2], m[3]);
            } else {
                // several documents, or the stream's end: one document after the other
                int a = 0;                                     // rows [a, b1) of the warp's 32
                for (int doc = fold_doc; doc < nd && a < 32; ++doc) {
                    const int b1 = s_off[doc + 1] - s0;
                    if (b1 <= a) continue;                     // (a slot without a document)
                    float m[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll
                    for (int jj = 0; jj < 4; ++jj)
                        if (sub + 8 * jj >= a && sub + 8 * jj < b1)
#pragma unroll
                            for (int e = 0; e < 4; ++e) m[e] = fmaxf(m[e], v[jj][e]);
                    publish(doc, m[0], m[1], m[2], m[3]);
                    a = b1;
                }
            }
        }
        cid = cid_next;
        cid_next = cid_far;
    }

    if (n_tiles == 0 && tid == 0 && !skip_loads) mbar_wait(bar_b, 0, wait_limit);   // never leave with the TMA load in flight
    tc_fence_before();
    __syncthreads();

    // ---- per document: add the per-query-token constant, sum over query tokens ----------------------------------------
    if (alive) {
        for (int dl = warp; dl < nd; dl += G4U_THREADS / 32) {
            const int32_t d = pruned[(int64_t)b * n_prune + j0 + dl];
            float v = 0.f;
            if (RQ) {                                   // fixed summation order: reproducible bits
                if (d >= 0 && lane == 0)
                    for (int i = 0; i < nq; ++i) v = __fadd_rn(v, f_unorder(docmax[dl * NQP + i]));
            } else if (d >= 0) {
                if (lane < nq) v = f_unorder(docmax[dl * NQP + lane]) * (1.0f / 16777216.0f) + kappa * s_sumq[lane];
                if (NQP > 32 && 32 + lane < nq) v += f_unorder(docmax[dl * NQP + 32 + lane]) * (1.0f / 16777216.0f) + kappa * s_sumq[32 + lane];
            }
            v = warp_sum(v);
            if (lane == 0) {
                float *out = score4 + (int64_t)b * n_prune + j0 + dl;
                *out = d >= 0 ? (q_base > 0 ? *out + v : v) : -INFINITY;      // (the first tokens' launch came before)
            }
        }
    }
    if (warp == 0) {
        tc_fence_after();
        tmem_dealloc(tmem, TMEM_COLS);
    }
}

template <int NQP, int NBITS, bool RQ>
static int launch_g4_umma(const Index &ix, const Params &p, int q_base, int nq, const float *queries, const int8_t *qdig4,
                          const int32_t *table, const int32_t *pruned, float *score4, uint32_t *status, cudaStream_t st)
{
    constexpr int N = 3 * NQP;
    const float delta = (ix.res_hi - ix.res_lo) / (float)(1 << ix.nbits);
    // RQ: the kappa slot carries c = 1 / (sqrt(D) * 2^22)
    const float kappa = RQ ? (float)(1.0 / (sqrt((double)ix.D) * 4194304.0)) : ix.res_lo + 0.5f * delta;
    CUtensorMap map_q;
    int rc = make_plane_map(&map_q, qdig4, (int64_t)p.B * residual_rows(p.nq), NQP);
    if (rc) return rc;
    // query planes, maxima
    size_t smem = 1024 + (size_t)N * 128 + sizeof(uint32_t) * G4U_MAX_DOCS * NQP + 32;
    // No more CTAs may become resident on an SM than its 512 tensor-memory columns serve: one more would sit in
    // tcgen05.alloc with its registers and shared memory until another leaves.  Registers cap the 128-column variants at
    // four or fewer and the 256-column ones at two; the latter ask for a third of an SM's shared memory plus one byte
    // besides, so that a build with fewer registers does not change that.
    if (N > 96 && smem < 227 * 1024 / 3 + 1) smem = 227 * 1024 / 3 + 1;
    const bool full = p.nq == NQP && nq == NQP;
    auto kern = full ? residual_maxsim_umma<NQP, NBITS, RQ, 128, true> : residual_maxsim_umma<NQP, NBITS, RQ, 128, false>;
    switch (ix.D) {                                          // (a multiple of 32 up to 128)
    case 32: kern = full ? residual_maxsim_umma<NQP, NBITS, RQ, 32, true> : residual_maxsim_umma<NQP, NBITS, RQ, 32, false>; break;
    case 64: kern = full ? residual_maxsim_umma<NQP, NBITS, RQ, 64, true> : residual_maxsim_umma<NQP, NBITS, RQ, 64, false>; break;
    case 96: kern = full ? residual_maxsim_umma<NQP, NBITS, RQ, 96, true> : residual_maxsim_umma<NQP, NBITS, RQ, 96, false>; break;
    }
    CHIMERA_CUDA(allow_shared(kern, smem));                  // (the same in every call of this kernel)
    // documents per CTA: whole waves of resident CTAs, as few as documents-per-CTA limit allows (a second wave of a few CTAs
    // costs as much as a full one: 37 queries of 777 survivors in 2.1 waves of 32 documents, or in three of 22)
    const int64_t slots = (int64_t)(NQP == 32 ? (RQ ? 4 : 3) : 2) * ix.sm_count, docs = (int64_t)p.n_prune * p.B;
    const int64_t waves = (docs + slots * G4U_MAX_DOCS - 1) / (slots * G4U_MAX_DOCS);
    int64_t per_query = waves * slots / p.B;               // CTAs per query
    if (per_query < 1) per_query = 1;
    int64_t dpc = (p.n_prune + per_query - 1) / per_query;
    if (dpc < 1) dpc = 1;
    if (dpc > G4U_MAX_DOCS) dpc = G4U_MAX_DOCS;
    dim3 grid((unsigned)((p.n_prune + dpc - 1) / dpc), (unsigned)p.B);
    const uint32_t *code_words = reinterpret_cast<const uint32_t *>(RQ ? ix.rq_bits : ix.codes);
    launch(kern, grid, 128 * (NQP / G4U_COLS), smem, st, map_q, queries, table, ix.K, nq, q_base, p.nq,
           residual_rows(p.nq), delta, kappa, pruned, p.n_prune, (int)dpc, ix.cids, code_words, ix.rq_inv, ix.doc_off, score4,
           status, wait_limit_cycles(), fault_skip_tma_loads());
    CHIMERA_CUDA(cudaGetLastError());
    count_launch(SLOT_G4);
    return CHIMERA_OK;
}

// More than 64 query tokens: the first 64, then the rest added to their scores (MMA N would exceed 256 with all of them).
template <int NBITS>
static int launch_g4_parts(const Index &ix, const Params &p, const float *queries, const int8_t *qdig4, const int32_t *table,
                           const int32_t *pruned, float *score4, uint32_t *status, cudaStream_t st)
{
    for (int q_base = 0; q_base < p.nq; q_base += 64) {
        const int nq = p.nq - q_base < 64 ? p.nq - q_base : 64;
        const int rc = nq <= 32 ? launch_g4_umma<32, NBITS, false>(ix, p, q_base, nq, queries, qdig4, table, pruned, score4, status, st)
                                : launch_g4_umma<64, NBITS, false>(ix, p, q_base, nq, queries, qdig4, table, pruned, score4, status, st);
        if (rc) return rc;
    }
    return CHIMERA_OK;
}

int launch_residual_scores_umma(const Index &ix, const Params &p, const float *queries, const int8_t *qdig4,
                                const int32_t *table, const int32_t *pruned, float *score4, uint32_t *status,
                                cudaStream_t st)
{
    return ix.nbits == 2 ? launch_g4_parts<2>(ix, p, queries, qdig4, table, pruned, score4, status, st)
                         : launch_g4_parts<1>(ix, p, queries, qdig4, table, pruned, score4, status, st);
}

// Complete 1-bit scores of the surviving documents on the RaBitQ codes; q_rot / qdig_rot belong to the rotated queries.
int launch_rabitq_scores_umma(const Index &ix, const Params &p, const float *q_rot, const int8_t *qdig_rot,
                              const int32_t *pruned, float *score4, uint32_t *status, cudaStream_t st)
{
    if (p.nq <= 32) return launch_g4_umma<32, 1, true>(ix, p, 0, p.nq, q_rot, qdig_rot, nullptr, pruned, score4, status, st);
    return launch_g4_umma<64, 1, true>(ix, p, 0, p.nq, q_rot, qdig_rot, nullptr, pruned, score4, status, st);
}

}  // namespace chimera
