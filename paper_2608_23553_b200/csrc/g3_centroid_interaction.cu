// Stage 3: centroid-interaction pruning.
//   CI(d) = sum_i max_{t in d} S[cid_t, i]      (the Chamfer aggregation rule of Sec. 4.2 -- per query token the
//                                                maximum over the document's tokens, then the sum over query
//                                                tokens -- applied to the centroid scores; integers, order-free)
//   keep the n_prune candidates with the largest CI, ties towards the smaller document id.
//
// Two phases when q_len is 32 or 64: cheap bounds lo(d) <= CI(d) <= hi(d) for every candidate from an 8-bit copy of
// the table (cand_range_kernel + ci_coarse_rng_kernel; ci_coarse_kernel for tables staged in shared memory and for
// corpora of 2^31 tokens or more), the documents whose hi reaches the n_prune-th largest lo (contender kernels), then
// exact CI (ci_wide_rng_kernel over the contenders' token ranges; ci_wide_kernel without ranges) and the exact
// selection among those only.  Other q_len: exact CI for every candidate
// (ci_kernel).
//
// ci_kernel: one warp per candidate document.  The document's centroid ids are streamed with coalesced 128-byte
// loads (lane = token), each is broadcast with a shuffle, and the warp gathers the table row S[cid, :] with
// lane = query token (one 128-byte line for 32 query tokens), keeping a running maximum per lane.
//
// select_kernel: one block per query.  Few of many: select_few.  Else radix select (11 + 11 + 10 bits) of the n_prune-th
// largest score, then an ordered compaction of the candidate list (which is ascending in id), so equal scores are resolved
// towards smaller ids and the survivors come out ascending.  With few queries per call the contender and selection steps run over 32
// blocks per query instead (contender_hist/count/write kernels, sels_* kernels), and shard_select_kernel merges the
// lists of a document-sharded search.
#include <limits.h>

#include "common.cuh"
#include "g3_select.cuh"

namespace chimera {

constexpr int CI_THREADS = 256;
constexpr int CI_WARPS = CI_THREADS / 32;

// Any q_len.  rng: NULL, or the documents' token ranges (first token, length); (CI, 0) stands for a document whose CI is
// known.  Instructions are the limit (21 a row, with a 64-bit product and a predicate for each, took 271 us for 8.3 million rows of 84
// bytes at 65 % of the issue rate), so a row's address is one 32 x 32-bit multiply-add and lanes past the last column read that one
// again instead of nothing.  The next 32 centroid ids are loaded ahead of the rows.
template <int NQW>   // 32-column groups handled per lane
__global__ void __launch_bounds__(CI_THREADS)
ci_kernel(const int32_t *__restrict__ table, int64_t K, int nq, const int32_t *__restrict__ cand,
          const int32_t *__restrict__ n_cand, int64_t maxc, const int32_t *__restrict__ cids,
          const int64_t *__restrict__ doc_off, const int2 *__restrict__ rng, int32_t *__restrict__ ci)
{
    pdl_entry();
    constexpr int U = NQW == 1 ? 16 : 8;                     // rows in flight (16 of short rows: 48 us where 8 take 63)
    const int b = blockIdx.y;
    const int lane = threadIdx.x & 31;
    const int n = n_cand[b];
    const char *col[NQW];                                    // this lane's columns of row 0
    const uint32_t row_bytes = 4u * (uint32_t)nq;
#pragma unroll
    for (int w = 0; w < NQW; ++w)
        col[w] = reinterpret_cast<const char *>(table + (int64_t)b * K * nq + (lane + 32 * w < nq ? lane + 32 * w : nq - 1));
    const int32_t *cb = cand + (int64_t)b * maxc;
    int32_t *out = ci + (int64_t)b * maxc;
    const int warps_per_query = gridDim.x * CI_WARPS;
    for (int j = blockIdx.x * CI_WARPS + (threadIdx.x >> 5); j < n; j += warps_per_query) {
        int64_t t0, t1;
        if (rng) {
            const int2 r = rng[(int64_t)b * maxc + j];
            if (r.y == 0) {
                if (lane == 0) out[j] = r.x;
                continue;
            }
            t0 = r.x;
            t1 = t0 + r.y;
        } else {
            const int64_t d = DBG_DOC(cb[j]);
            t0 = doc_off[d];
            t1 = doc_off[d + 1];
        }
        int m[NQW];
#pragma unroll
        for (int w = 0; w < NQW; ++w) m[w] = INT_MIN;
        // lanes past the end repeat the last token: a duplicate cannot change a maximum
        int32_t next = t0 < t1 ? cids[t0 + lane < t1 ? t0 + lane : t1 - 1] : 0;
        for (int64_t base = t0; base < t1; base += 32) {
            const int cnt = (int)((t1 - base) < 32 ? (t1 - base) : 32);
            const int32_t cidv = next;
            if (base + 32 < t1) next = cids[base + 32 + lane < t1 ? base + 32 + lane : t1 - 1];
            for (int t = 0; t < cnt; t += U) {
                int32_t v[U][NQW];
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const uint32_t c = (uint32_t)DBG_CID(__shfl_sync(0xffffffffu, cidv, t + u));       // t + u <= 31
#pragma unroll
                    for (int w = 0; w < NQW; ++w)
                        v[u][w] = __ldg(reinterpret_cast<const int32_t *>(col[w] + (uint64_t)c * row_bytes));
                }
#pragma unroll
                for (int u = 0; u < U; u += 2)
#pragma unroll
                    for (int w = 0; w < NQW; ++w) m[w] = __vimax3_s32(m[w], v[u][w], v[u + 1][w]);
            }
        }
        int s = 0;
#pragma unroll
        for (int w = 0; w < NQW; ++w)
            if (lane + 32 * w < nq) s += m[w];
        s = warp_sum(s);
        if (lane == 0) out[j] = s;
    }
}

// Wide variant for q_len = 4 * LPR (LPR = 8 or 16 lanes per table row): every lane loads 16 bytes (four query
// tokens) of a row, so one load instruction of the warp covers 32 / LPR document tokens.  Lane group g = lane / LPR
// takes tokens g, g + TPL, g + 2 TPL, ... of each 32-token slab; the group maxima are merged with shuffles at the end.
template <int LPR>
__global__ void __launch_bounds__(CI_THREADS)
ci_wide_kernel(const int32_t *__restrict__ table, int64_t K, const int32_t *__restrict__ cand,
               const int32_t *__restrict__ n_cand, int64_t maxc, const int32_t *__restrict__ cids,
               const int64_t *__restrict__ doc_off, int32_t *__restrict__ ci)
{
    pdl_entry();
    constexpr int NQ = 4 * LPR;
    constexpr int TPL = 32 / LPR;                 // tokens per warp-wide load
    constexpr int UNROLL = 8;
    const int b = blockIdx.y;
    const int lane = threadIdx.x & 31;
    const int grp = lane / LPR, sub = lane % LPR;
    const int n = n_cand[b];
    const int4 *tb = reinterpret_cast<const int4 *>(table + (int64_t)b * K * NQ) + sub;
    const int32_t *cb = cand + (int64_t)b * maxc;
    int32_t *out = ci + (int64_t)b * maxc;
    const int warps_per_query = gridDim.x * CI_WARPS;
    for (int j = blockIdx.x * CI_WARPS + (threadIdx.x >> 5); j < n; j += warps_per_query) {
        const int64_t d = DBG_DOC(cb[j]);
        const int64_t t0 = doc_off[d], t1 = doc_off[d + 1];
        int4 m = make_int4(INT_MIN, INT_MIN, INT_MIN, INT_MIN);
        for (int64_t base = t0; base < t1; base += 32) {
            const int cnt = (int)((t1 - base) < 32 ? (t1 - base) : 32);
            // lanes past the end repeat the last token: a duplicate cannot change a maximum
            const int32_t cidv = cids[base + (lane < cnt ? lane : cnt - 1)];
            for (int s = 0; s * TPL < cnt; s += UNROLL) {
                int4 v[UNROLL];
#pragma unroll
                for (int u = 0; u < UNROLL; ++u) {
                    int src = (s + u) * TPL + grp;
                    src = src < 32 ? src : 31;    // lane 31 holds a valid (possibly repeated) token
                    const int32_t c = __shfl_sync(0xffffffffu, cidv, src);
                    v[u] = __ldg(tb + (int64_t)DBG_CID(c) * LPR);
                }
#pragma unroll
                for (int u = 0; u < UNROLL; u += 2) {          // three-input integer maximum: two rows per instruction
                    m.x = __vimax3_s32(m.x, v[u].x, v[u + 1].x);
                    m.y = __vimax3_s32(m.y, v[u].y, v[u + 1].y);
                    m.z = __vimax3_s32(m.z, v[u].z, v[u + 1].z);
                    m.w = __vimax3_s32(m.w, v[u].w, v[u + 1].w);
                }
            }
        }
        // merge the TPL lane groups (same columns, different tokens)
#pragma unroll
        for (int o = LPR; o < 32; o <<= 1) {
            m.x = max(m.x, __shfl_xor_sync(0xffffffffu, m.x, o));
            m.y = max(m.y, __shfl_xor_sync(0xffffffffu, m.y, o));
            m.z = max(m.z, __shfl_xor_sync(0xffffffffu, m.z, o));
            m.w = max(m.w, __shfl_xor_sync(0xffffffffu, m.w, o));
        }
        // sum over the NQ columns: four per lane, LPR lanes
        int sum = m.x + m.y + m.z + m.w;
#pragma unroll
        for (int o = LPR >> 1; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
        if (lane == 0) out[j] = sum;
    }
}

// The wide variant over precomputed token ranges (first token, length) of the documents to score: a warp owns a
// contiguous run of them and takes them 32 at a time -- one coalesced load of the ranges, handed out by shuffle -- instead of the
// dependent chain id -> offsets -> centroid ids per document.  Latency is the limit (79 % of the stalls; a third of the rows come
// from DRAM), so the next 32 centroid ids, of this document or the next, are always on their way while rows are looked up: Mid,
// batch 256, 1,077 -> 1,041 us; 512-token documents, 64 queries of 64 tokens, 1,951 -> 1,792.  32 bytes a lane instead of 16 are
// no faster (1,097, 1,834), and rows that L1 does not keep much slower (1,440).
template <int LPR>
__global__ void __launch_bounds__(CI_THREADS)
ci_wide_rng_kernel(const int32_t *__restrict__ table, int64_t K, const int2 *__restrict__ rng,
                   const int32_t *__restrict__ n_docs, int64_t maxc, const int32_t *__restrict__ cids,
                   int32_t *__restrict__ ci)
{
    pdl_entry();
    constexpr int NQ = 4 * LPR;
    constexpr int TPL = 32 / LPR;                 // tokens per warp-wide load
    constexpr int UNROLL = 8;
    const int b = blockIdx.y;
    const int lane = threadIdx.x & 31;
    const int grp = lane / LPR, sub = lane % LPR;
    const int n = n_docs[b];
    const int4 *tb = reinterpret_cast<const int4 *>(table + (int64_t)b * K * NQ) + sub;
    const int2 *rb = rng + (int64_t)b * maxc;
    int32_t *out = ci + (int64_t)b * maxc;
    const int warps_per_query = gridDim.x * CI_WARPS;
    const int per_warp = (n + warps_per_query - 1) / warps_per_query;
    const int wq = blockIdx.x * CI_WARPS + (threadIdx.x >> 5);
    const int j_begin = wq * per_warp < n ? wq * per_warp : n;
    const int j_end = j_begin + per_warp < n ? j_begin + per_warp : n;
    for (int jb = j_begin; jb < j_end; jb += 32) {
        const int cnt_docs = j_end - jb < 32 ? j_end - jb : 32;
        int2 mine = lane < cnt_docs ? rb[jb + lane] : make_int2(0, 1);
        int my_sum = 0;
        if (mine.y == 0) {                                 // its CI is known and passes through
            my_sum = mine.x;
            mine.x = 0;
        }
        int32_t nx_cid;
        {
            const int t0 = __shfl_sync(0xffffffffu, mine.x, 0), len = __shfl_sync(0xffffffffu, mine.y, 0);
            nx_cid = cids[DBG_TOK((int64_t)t0 + (lane < len - 1 ? lane : len > 0 ? len - 1 : 0))];
        }
        for (int di = 0; di < cnt_docs; ++di) {
            const int t0 = __shfl_sync(0xffffffffu, mine.x, di), len = __shfl_sync(0xffffffffu, mine.y, di);
            const int n0 = __shfl_sync(0xffffffffu, mine.x, di + 1 < cnt_docs ? di + 1 : di);
            const int nl = __shfl_sync(0xffffffffu, mine.y, di + 1 < cnt_docs ? di + 1 : di);
            int4 m = make_int4(INT_MIN, INT_MIN, INT_MIN, INT_MIN);
            for (int base = 0; base < len || base == 0; base += 32) {
                const int cnt = len - base < 32 ? len - base : 32;
                // the next 32 ids, of this document or the next one, travel with the rows of these; lanes past the end repeat the
                // last token: a duplicate cannot change a maximum
                const int32_t cidv = nx_cid;
                {
                    const bool more = base + 32 < len;
                    const int64_t f0 = more ? (int64_t)t0 + base + 32 : n0;
                    const int fl = more ? len - base - 32 : nl;
                    nx_cid = cids[DBG_TOK(f0 + (lane < fl - 1 ? lane : fl > 0 ? fl - 1 : 0))];
                }
                for (int s = 0; s * TPL < cnt; s += UNROLL) {
                    int4 v[UNROLL];
#pragma unroll
                    for (int u = 0; u < UNROLL; ++u) {
                        int src = (s + u) * TPL + grp;
                        src = src < 32 ? src : 31;    // lane 31 holds a valid (possibly repeated) token
                        const int32_t c = __shfl_sync(0xffffffffu, cidv, src);
                        v[u] = __ldg(tb + (int64_t)DBG_CID(c) * LPR);
                    }
#pragma unroll
                    for (int u = 0; u < UNROLL; u += 2) {
                        m.x = __vimax3_s32(m.x, v[u].x, v[u + 1].x);
                        m.y = __vimax3_s32(m.y, v[u].y, v[u + 1].y);
                        m.z = __vimax3_s32(m.z, v[u].z, v[u + 1].z);
                        m.w = __vimax3_s32(m.w, v[u].w, v[u + 1].w);
                    }
                }
            }
            if (len == 0) continue;
#pragma unroll
            for (int o = LPR; o < 32; o <<= 1) {           // merge the TPL lane groups
                m.x = max(m.x, __shfl_xor_sync(0xffffffffu, m.x, o));
                m.y = max(m.y, __shfl_xor_sync(0xffffffffu, m.y, o));
                m.z = max(m.z, __shfl_xor_sync(0xffffffffu, m.z, o));
                m.w = max(m.w, __shfl_xor_sync(0xffffffffu, m.w, o));
            }
            int sum = m.x + m.y + m.z + m.w;
#pragma unroll
            for (int o = LPR >> 1; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
            sum = __shfl_sync(0xffffffffu, sum, 0);
            if (lane == di) my_sum = sum;
        }
        if (lane < cnt_docs) out[jb + lane] = my_sum;
    }
}

// ------------------------------------------------------------------------------------------------ coarse bounds --
// Bounds on CI from the 8-bit table U8[c, i] = clamp(S[c, i] >> 16, 0, 255) (stage 1 writes it next to the exact
// table): 256 buckets of width 2^16 over [0, 2^24), everything negative in bucket 0, everything from 255 * 2^16 up in
// bucket 255.  |S| <= 2^24 + 2^16 = SMAX: queries and centroids are at most unit-norm up to 2^-10 (checked where their
// fixed-point digits are made; a longer row is reported through the status word).  The map is monotone, so
// m_i = max_t U8[cid_t, i] is the bucket of the exact maximum:
//     2^16 m_i <= max_t S <= 2^16 m_i + 2^16 - 1        for 0 < m_i < 255,
// the lower end drops to -SMAX for m_i = 0 and the upper end rises to SMAX = 2^16 * 255 + 2^17 for m_i = 255.  With
// sum = sum_i m_i, zeros = #{i : m_i = 0}, sat = #{i : m_i = 255}:
//     lo(d) = 2^16 sum - zeros SMAX  <=  CI(d)  <=  2^16 sum + nq (2^16 - 1) + (2^16 + 1) sat = hi(d).
// (The scores that decide a maximum are positive -- a document token close to the query token -- so the buckets are
// spent on [0, 1) and a column whose best score is negative only loosens lo.)  A row of U8 is q_len bytes -- one
// 32-byte sector for 32 query
// tokens instead of four -- and a lane's 16-byte load covers 16 query tokens, so one warp load covers 32 / LPR tokens
// (LPR = q_len / 16 lanes per row).  The running maxima fold two rows per instruction with the three-input packed
// 16-bit integer maximum (see coarse_accumulate2).
// packed = sum | sat << 16 | zeros << 24 (see above)
__device__ __forceinline__ int32_t coarse_lo(int packed)
{
    return ((packed & 0xffff) << 16) - (packed >> 24) * ((1 << 24) + (1 << 16));
}
__device__ __forceinline__ int32_t coarse_hi(int packed, int nq)
{
    return ((packed & 0xffff) << 16) + nq * ((1 << 16) - 1) + ((packed >> 16) & 0xff) * ((1 << 16) + 1);
}
// Running maxima of a lane's 16 columns in eight registers of two 16-bit fields each, updated from two rows at a time
// with the three-input packed 16-bit maximum.  A field compares as (column byte << 8 | whatever lies below it), so the
// winner's HIGH byte is the column's maximum and no widening is needed: the odd bytes of a word already sit in the high
// byte of a field (registers 4..7 take the raw words), the even bytes get there with one shift (registers 0..3).
// coarse_field() extracts a field's maximum at the end.
__device__ __forceinline__ void coarse_accumulate2(uint32_t (&m)[8], const int4 &va, const int4 &vb)
{
    const uint32_t a[4] = {(uint32_t)va.x, (uint32_t)va.y, (uint32_t)va.z, (uint32_t)va.w};
    const uint32_t b[4] = {(uint32_t)vb.x, (uint32_t)vb.y, (uint32_t)vb.z, (uint32_t)vb.w};
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        m[k] = __vimax3_u16x2(m[k], a[k] << 8, b[k] << 8);
        m[4 + k] = __vimax3_u16x2(m[4 + k], a[k], b[k]);
    }
}
__device__ __forceinline__ int coarse_field_lo(uint32_t m) { return (int)((m >> 8) & 0xffu); }
__device__ __forceinline__ int coarse_field_hi(uint32_t m) { return (int)(m >> 24); }
// cut: of a call that may cut (kept not NULL): nothing is done when it does.
// SMEM = true: the query's whole 8-bit table (K * q_len bytes) is first staged in shared memory and the row lookups
// are shared-memory loads (small K only); blocks are then larger (THREADS) because only one fits an SM.
template <int LPR, bool SMEM, int THREADS>
__global__ void __launch_bounds__(THREADS)
ci_coarse_kernel(const uint8_t *__restrict__ table8, int64_t K, const int32_t *__restrict__ cand,
                 const int32_t *__restrict__ n_cand, int64_t maxc, const int32_t *__restrict__ cids,
                 const int64_t *__restrict__ doc_off, int32_t *__restrict__ lo, int32_t *__restrict__ hi,
                 FirstCut cut)
{
    pdl_entry();
    if (cut.kept && cut.on()) return;             // (the scan over ranges does it)
    extern __shared__ int4 smem_table[];
    constexpr int WARPS = THREADS / 32;
    constexpr int NQ = 16 * LPR;
    constexpr int TPL = 32 / LPR;                 // tokens per warp-wide load
    constexpr int STEPS = 32 / TPL;               // loads per 32-token slab (= LPR)
    constexpr int SLABS = 2;                      // 32-token slabs per iteration (more costs occupancy and loses)
    const int b = blockIdx.y;
    const int lane = threadIdx.x & 31;
    const int grp = lane / LPR, sub = lane % LPR;
    const int n = n_cand[b];
    const int4 *tb = reinterpret_cast<const int4 *>(table8 + (int64_t)b * K * NQ) + sub;
    if (SMEM) {
        const int4 *src = reinterpret_cast<const int4 *>(table8 + (int64_t)b * K * NQ);
        for (int64_t e = threadIdx.x; e < K * LPR; e += THREADS) smem_table[e] = __ldg(src + e);
        __syncthreads();
    }
    const int4 *ts = smem_table + sub;
    const int32_t *cb = cand + (int64_t)b * maxc;
    const int warps_per_query = gridDim.x * WARPS;
    // The chain candidate id -> token range -> first centroid ids is three dependent loads: it is issued one document
    // ahead, so it overlaps the row gathers of the current document.
    int64_t nx_t0 = 0, nx_t1 = 0;
    int32_t nx_cid[SLABS];
    auto prefetch = [&](int j) {
        const int64_t d = DBG_DOC(cb[j]);
        nx_t0 = doc_off[d];
        nx_t1 = doc_off[d + 1];
#pragma unroll
        for (int k = 0; k < SLABS; ++k) {
            const int64_t i = nx_t0 + 32 * k + lane;
            nx_cid[k] = cids[i < nx_t1 - 1 ? i : nx_t1 - 1];
        }
    };
    int j = blockIdx.x * WARPS + (threadIdx.x >> 5);
    if (j < n) prefetch(j);
    for (; j < n; j += warps_per_query) {
        const int64_t t0 = nx_t0, t1 = nx_t1;
        int32_t cid[SLABS];
#pragma unroll
        for (int k = 0; k < SLABS; ++k) cid[k] = nx_cid[k];
        if (j + warps_per_query < n) prefetch(j + warps_per_query);
        uint32_t m[8];
#pragma unroll
        for (int r = 0; r < 8; ++r) m[r] = 0u;
        for (int64_t base = t0; base < t1; base += 32 * SLABS) {
            // up to SLABS 32-token slabs per iteration, all their row loads in flight together; lanes past the end
            // repeat the last token (harmless for a maximum)
            if (base != t0) {
                const int64_t last = t1 - 1;
#pragma unroll
                for (int k = 0; k < SLABS; ++k) {
                    const int64_t i = base + 32 * k + lane;
                    cid[k] = cids[i < last ? i : last];
                }
            }
            int4 v[SLABS * STEPS];
#pragma unroll
            for (int k = 0; k < SLABS; ++k) {
                if (k == 0 || base + 32 * k < t1) {
#pragma unroll
                    for (int s = 0; s < STEPS; ++s) {
                        const int32_t c = __shfl_sync(0xffffffffu, cid[k], s * TPL + grp);
                        v[k * STEPS + s] = SMEM ? ts[DBG_CID(c) * LPR] : __ldg(tb + (int64_t)DBG_CID(c) * LPR);
                    }
                }
            }
#pragma unroll
            for (int k = 0; k < SLABS; ++k) {
                if (k == 0 || base + 32 * k < t1) {
#pragma unroll
                    for (int s = 0; s < STEPS; s += 2) coarse_accumulate2(m, v[k * STEPS + s], v[k * STEPS + s + 1]);
                }
            }
        }
        // Merge the lane groups (same columns, different tokens).  While a lane still holds several registers each
        // exchange keeps one half of them and hands the other half to the partner, so the data halves per step;
        // the remaining steps exchange the last register whole (those lanes end up with duplicates).
        int nreg = 8;
        uint32_t dup_mask = 0;
#pragma unroll
        for (int o = 16; o >= LPR; o >>= 1) {
            if (nreg > 1) {
                const int half = nreg >> 1;
                const bool up = (lane & o) != 0;
#pragma unroll
                for (int r = 0; r < 4; ++r) {
                    if (r < half) {
                        const uint32_t send = up ? m[r] : m[r + half];
                        const uint32_t keep = up ? m[r + half] : m[r];
                        m[r] = __vmaxu2(keep, __shfl_xor_sync(0xffffffffu, send, o));
                    }
                }
                nreg = half;
            } else {
                m[0] = __vmaxu2(m[0], __shfl_xor_sync(0xffffffffu, m[0], o));
                dup_mask |= (uint32_t)o;
            }
        }
        // every lane now holds the maxima of two columns; sum over columns (skipping duplicate lanes)
        const int u_lo = coarse_field_lo(m[0]), u_hi = coarse_field_hi(m[0]);
        int packed = 0;                                         // sum of maxima | saturated << 16 | zeros << 24
        if ((lane & dup_mask) == 0)
            packed = (u_lo + u_hi) + (((u_lo >= 255) + (u_hi >= 255)) << 16) + (((u_lo == 0) + (u_hi == 0)) << 24);
        packed = __reduce_add_sync(0xffffffffu, packed);        // sum <= 255 * 64 < 2^16, counts <= 64
        if (lane == 0) {
            lo[(int64_t)b * maxc + j] = coarse_lo(packed);
            hi[(int64_t)b * maxc + j] = coarse_hi(packed, NQ);
        }
    }
}

// Token range (first token, length) of every candidate, written once per search: the scan then finds a document's
// tokens with one coalesced load per 32 documents instead of the dependent chain id -> offsets per document.
__global__ void __launch_bounds__(256)
cand_range_kernel(const int32_t *__restrict__ cand, const int32_t *__restrict__ n_cand, int64_t maxc,
                  const int64_t *__restrict__ doc_off, int2 *__restrict__ rng, int32_t *__restrict__ cont_hist)
{
    pdl_entry();
    const int b = blockIdx.y;
    if (cont_hist)                                        // the contender step's histogram (at the head of its scratch row)
        for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < CONT_BINS; i += gridDim.x * blockDim.x)
            cont_hist[(int64_t)b * maxc + i] = 0;
    const int n = n_cand[b];
    for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < n; j += gridDim.x * blockDim.x) {
        const int64_t d = DBG_DOC(cand[(int64_t)b * maxc + j]);
        const int64_t t0 = doc_off[d];
        rng[(int64_t)b * maxc + j] = make_int2((int)t0, (int)(doc_off[d + 1] - t0));
    }
}

// The bound scan over precomputed token ranges (corpora with fewer than 2^31 tokens).  A warp owns a contiguous run of
// the query's candidates and takes them 32 at a time: lane i loads the range of document i of the group (one coalesced
// load), the ranges are handed out by shuffle, and while document i is scanned the first centroid ids of document
// i + 1 are already being fetched -- a one-level prefetch where the per-document chain used to have three levels.
// The 32 results of a group are written back coalesced.
// nq: the columns that count; those up to 16 LPR are zero in every row.  list (may be NULL): the places of the ranges to take.
// lo may be NULL (and has to be where nq < 16 LPR).
template <int LPR>
__device__ __forceinline__ void
ci_coarse_rng_body(const uint8_t *__restrict__ table8, int64_t K, int nq, const int2 *__restrict__ rng,
                     const int32_t *__restrict__ list, const int32_t *__restrict__ n_cand, int64_t maxc, const int32_t *__restrict__ cids,
                     int32_t *__restrict__ lo, int32_t *__restrict__ hi)
{
    constexpr int NQ = 16 * LPR;
    constexpr int TPL = 32 / LPR;                 // tokens per warp-wide load
    constexpr int STEPS = 32 / TPL;               // loads per 32-token slab (= LPR)
    // 32-token slabs per iteration, and whether the centroid ids of the document after next are pulled into L2.
    // Measured (bound scan, batch 256): for 32-byte rows one slab without that prefetch is the fastest of the four
    // combinations (Mid 14.21 ms against 14.45 ms for two slabs with it, 14.54 / 14.75 ms for the mixed ones; Large
    // 28.2 against 28.7 ms); for 64-byte rows two slabs with the prefetch are (long documents: 28.8 against 29.1 ms).
    constexpr int SLABS = LPR == 4 ? 2 : 1;
    constexpr bool PREFETCH_L2 = LPR == 4;
    const int b = blockIdx.y;
    const int lane = threadIdx.x & 31;
    const int grp = lane / LPR, sub = lane % LPR;
    const int n = n_cand[b];
    const int4 *tb = reinterpret_cast<const int4 *>(table8 + (int64_t)b * K * NQ) + sub;
    const int2 *rb = rng + (int64_t)b * maxc;
    const int warps_per_query = gridDim.x * CI_WARPS;
    const int per_warp = (n + warps_per_query - 1) / warps_per_query;
    const int wq = blockIdx.x * CI_WARPS + (threadIdx.x >> 5);
    const int j_begin = wq * per_warp < n ? wq * per_warp : n;
    const int j_end = j_begin + per_warp < n ? j_begin + per_warp : n;

    for (int jb = j_begin; jb < j_end; jb += 32) {
        const int cnt = j_end - jb < 32 ? j_end - jb : 32;
        const int place = lane >= cnt ? 0 : list ? list[(int64_t)b * maxc + jb + lane] : jb + lane;
        int2 mine = lane < cnt ? rb[place] : make_int2(0, 1);
        int my_lo = 0, my_hi = 0;
        if (mine.y == 0) {                             // its exact CI is known: both bounds
            my_lo = my_hi = mine.x;
            mine.x = 0;
        }
        int32_t nx_cid[SLABS];
        {
            const int t0 = __shfl_sync(0xffffffffu, mine.x, 0), len = __shfl_sync(0xffffffffu, mine.y, 0);
#pragma unroll
            for (int k = 0; k < SLABS; ++k) {
                const int i = 32 * k + lane;
                nx_cid[k] = cids[DBG_TOK((int64_t)t0 + (i < len - 1 ? i : len > 0 ? len - 1 : 0))];
            }
        }
        for (int di = 0; di < cnt; ++di) {
            const int t0 = __shfl_sync(0xffffffffu, mine.x, di), len = __shfl_sync(0xffffffffu, mine.y, di);
            int32_t cid[SLABS];
#pragma unroll
            for (int k = 0; k < SLABS; ++k) cid[k] = nx_cid[k];
            if (PREFETCH_L2 && di + 2 < cnt) {         // two documents ahead: pull the centroid ids into L2
                const int p0 = __shfl_sync(0xffffffffu, mine.x, di + 2), pl = __shfl_sync(0xffffffffu, mine.y, di + 2);
                if (lane * 32 < pl) asm volatile("prefetch.global.L2 [%0];" ::"l"(cids + (int64_t)p0 + lane * 32));
            }
            if (di + 1 < cnt) {
                const int n0 = __shfl_sync(0xffffffffu, mine.x, di + 1), nl = __shfl_sync(0xffffffffu, mine.y, di + 1);
#pragma unroll
                for (int k = 0; k < SLABS; ++k) {
                    const int i = 32 * k + lane;
                    nx_cid[k] = cids[DBG_TOK((int64_t)n0 + (i < nl - 1 ? i : nl > 0 ? nl - 1 : 0))];
                }
            }
            if (len == 0) continue;
            uint32_t m[8];
#pragma unroll
            for (int r = 0; r < 8; ++r) m[r] = 0u;
            for (int base = 0; base < len; base += 32 * SLABS) {
                // lanes past the end repeat the last token (harmless for a maximum)
                int4 v[SLABS * STEPS];
#pragma unroll
                for (int k = 0; k < SLABS; ++k) {
                    if (k == 0 || base + 32 * k < len) {
#pragma unroll
                        for (int s = 0; s < STEPS; ++s) {
                            const int32_t c = __shfl_sync(0xffffffffu, cid[k], s * TPL + grp);
                            v[k * STEPS + s] = __ldg(tb + (int64_t)DBG_CID(c) * LPR);
                        }
                    }
                }
                // the centroid ids of the next iteration travel while this iteration's rows do
                if (base + 32 * SLABS < len) {
#pragma unroll
                    for (int k = 0; k < SLABS; ++k) {
                        const int i = base + 32 * SLABS + 32 * k + lane;
                        cid[k] = cids[DBG_TOK((int64_t)t0 + (i < len - 1 ? i : len - 1))];
                    }
                }
#pragma unroll
                for (int k = 0; k < SLABS; ++k) {
                    if (k == 0 || base + 32 * k < len) {
#pragma unroll
                        for (int s = 0; s < STEPS; s += 2)
                            coarse_accumulate2(m, v[k * STEPS + s], v[k * STEPS + s + 1]);
                    }
                }
            }
            // merge the lane groups (same columns, different tokens): each exchange keeps one half of the registers
            int nreg = 8;
            uint32_t dup_mask = 0;
#pragma unroll
            for (int o = 16; o >= LPR; o >>= 1) {
                if (nreg > 1) {
                    const int half = nreg >> 1;
                    const bool up = (lane & o) != 0;
#pragma unroll
                    for (int r = 0; r < 4; ++r) {
                        if (r < half) {
                            const uint32_t send = up ? m[r] : m[r + half];
                            const uint32_t keep = up ? m[r + half] : m[r];
                            m[r] = __vmaxu2(keep, __shfl_xor_sync(0xffffffffu, send, o));
                        }
                    }
                    nreg = half;
                } else {
                    m[0] = __vmaxu2(m[0], __shfl_xor_sync(0xffffffffu, m[0], o));
                    dup_mask |= (uint32_t)o;
                }
            }
            int packed = 0;                                         // sum of maxima | saturated << 16 | zeros << 24
#pragma unroll
            for (int r = 0; r < (LPR == 8 ? 2 : 1); ++r) {
                const int u_lo = coarse_field_lo(m[r]), u_hi = coarse_field_hi(m[r]);
                if ((lane & dup_mask) == 0)
                    packed += (u_lo + u_hi) + (((u_lo >= 255) + (u_hi >= 255)) << 16) +
                              (LPR == 8 ? 0 : ((u_lo == 0) + (u_hi == 0)) << 24);
            }
            packed = __reduce_add_sync(0xffffffffu, packed);
            if (lane == di) {                                       // lane di keeps the result of document di
                my_lo = coarse_lo(packed);
                my_hi = coarse_hi(packed, nq);
            }
        }
        if (lane < cnt) {
            if (lo) lo[(int64_t)b * maxc + place] = my_lo;
            hi[(int64_t)b * maxc + place] = my_hi;
        }
    }
}

// cut: of a call that may cut (kept not NULL): nothing is done when it does (ci_bound_kernel has the bounds then).
// Four blocks per SM, that is 64 registers: 64-byte rows would take 75 (long-document corpus: 27.1 against 28.4 ms), 32-byte rows
// 48, with fewer loads in flight (one query, 190,000 documents: 219 against 245 us).
template <int LPR>
__global__ void __launch_bounds__(CI_THREADS, 4)
ci_coarse_rng_kernel(const uint8_t *__restrict__ table8, int64_t K, const int2 *__restrict__ rng,
                     const int32_t *__restrict__ n_cand, int64_t maxc, const int32_t *__restrict__ cids,
                     int32_t *__restrict__ lo, int32_t *__restrict__ hi, FirstCut cut)
{
    pdl_entry();
    if (cut.kept && cut.on()) return;
    ci_coarse_rng_body<LPR>(table8, K, 16 * LPR, rng, nullptr, n_cand, maxc, cids, lo, hi);
}
// Upper bounds of what the first cut keeps, from the rows of few tokens.  A centroid counts as near when its score reaches
// theta_i for some query token i (mask: a bit per centroid).  The others cannot raise a column's maximum above theta_i, so
//     CI(d) <= sum_i max(theta_i, max over the near tokens of S[c_t, i]),
// and a fifth of the tokens are near (120 tokens, 32 columns, about one token above each threshold).  Documents whose bound
// reaches tau, one in six, go on to ci_rest_kernel.
// Measured (all kept documents at once / both kernels): Mid, batch 256, 1,717 us / 988 + 385; 512-token documents, 64 queries of
// 64 tokens, 1,795 / 856 + 223; 262,144 centroids, batch 256, 4,458 / 2,724 + 1,034.
// With few rows left to look up the instructions around them count (a document per warp: 1,890 us, 570 instructions each), so four
// documents share a warp, eight lanes each, those of a group of 32 taken by length: a bit per token from shared memory says
// whether it is near, near ids are collected in shared memory and their rows looked up 8 / LPR at a time and document.  nq: the columns that count; the rest of
// the 16 LPR are zero in every row.  Byte x of a row is column x / RUNS + 32 (x % RUNS), or x where stage 1 wrote the rows (RUNS as an
// argument: 1,013 us where constants take 981, Mid, batch 256).  rng: token ranges; (CI, 0) stands for a document whose CI is known.
constexpr int BOUND_THREADS = 512;
constexpr int BOUND_LIST = 64, BOUND_PITCH = BOUND_LIST + 8;
template <int LPR>
__global__ void __launch_bounds__(BOUND_THREADS, 2)
ci_bound_kernel(const uint8_t *__restrict__ table8, int64_t K, int nq, const uint32_t *__restrict__ mask, int mask_words,
                const int32_t *__restrict__ theta, const int32_t *__restrict__ tau, const int2 *__restrict__ rng,
                const int32_t *__restrict__ n_docs, int64_t maxc, const int32_t *__restrict__ cids, int32_t *__restrict__ hi,
                int32_t *__restrict__ rest, int32_t *__restrict__ n_rest, FirstCut cut)
{
    pdl_entry();
    constexpr int NQ = 16 * LPR, RPS = 8 / LPR;              // columns of a row, rows per step and document
    constexpr int RUNS = NQ / 32;                            // of a row that the first cut made (stage 1: nq == NQ, in order)
    constexpr int NF = LPR;                                  // registers (two columns each) of a lane after the folding
    constexpr int U = 4;                                     // steps in flight
    extern __shared__ uint32_t s_mask[];                     // and a zero word for positions past a document's end
    __shared__ int32_t s_ids[BOUND_THREADS / 32][4][BOUND_PITCH];
    __shared__ int32_t s_res[BOUND_THREADS / 32][32];
    __shared__ uint8_t s_ord[BOUND_THREADS / 32][32];
    const bool on = cut.on();
    const int b = blockIdx.y, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int dg = lane >> 3, l8 = lane & 7, grp = l8 / LPR, sub = l8 % LPR;
    const int n = n_docs[b];
    const int warps_per_query = gridDim.x * (BOUND_THREADS / 32);
    const int per_warp = (n + warps_per_query - 1) / warps_per_query;
    if (!on || (int)blockIdx.x * (BOUND_THREADS / 32) * per_warp >= n) return;
    for (int i = threadIdx.x; i <= mask_words; i += BOUND_THREADS)
        s_mask[i] = i == mask_words ? 0u : __ldg(mask + (int64_t)b * mask_words + i);
    const int32_t nobody = 32 * mask_words, limit = tau[b];
    const int4 *tb = reinterpret_cast<const int4 *>(table8 + (int64_t)b * K * NQ) + sub;
    // the fields (see coarse_accumulate2) that this lane holds after the folding, with theta - 1 in the columns
    uint32_t floor_f[8];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        uint32_t w = 0;
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const int at = 16 * sub + 4 * k + e, col = nq == NQ ? at : at / RUNS + 32 * (at % RUNS);
            if (col < nq) w |= (uint32_t)(theta[(int64_t)b * nq + col] - 1) << (8 * e);
        }
        floor_f[k] = w << 8;
        floor_f[4 + k] = w;
    }
    {
        int nreg = 8;
#pragma unroll
        for (int o = 4; o >= LPR; o >>= 1) {
            nreg >>= 1;
#pragma unroll
            for (int r = 0; r < 4; ++r)
                if (r < nreg && (l8 & o)) floor_f[r] = floor_f[r + nreg];
        }
    }
    __syncthreads();
    int32_t *ids = s_ids[warp][dg];
    const int2 *rb = rng + (int64_t)b * maxc;
    const int wq = blockIdx.x * (BOUND_THREADS / 32) + warp;
    const int j_begin = wq * per_warp < n ? wq * per_warp : n;
    const int j_end = j_begin + per_warp < n ? j_begin + per_warp : n;
    for (int jb = j_begin; jb < j_end; jb += 32) {
        const int cnt_docs = j_end - jb < 32 ? j_end - jb : 32;
        const int2 mine = lane < cnt_docs ? rb[jb + lane] : make_int2(0, 0);
        // longest first; documents whose CI is known (no tokens) come last and are not looked at
        const int key = mine.y << 5 | lane;
        int rank = 0;
#pragma unroll
        for (int i = 0; i < 32; ++i) rank += __shfl_sync(0xffffffffu, key, i) > key ? 1 : 0;
        __syncwarp();
        s_ord[warp][rank] = (uint8_t)lane;
        s_res[warp][lane] = mine.x;
        __syncwarp();
        const int todo = __popc(__ballot_sync(0xffffffffu, mine.y > 0));
        // ids of positions from ... from + 31 of the group's document, `nobody` past its end
        int32_t id[4];
        auto load_ids = [&](int t0, int from, int len) {
            const int32_t *src = cids + DBG_TOK((int64_t)(len > 0 ? t0 : 0)) + from + l8;
#pragma unroll
            for (int k = 0; k < 4; ++k) id[k] = from + l8 + 8 * k < len ? DBG_CID(__ldg(src + 8 * k)) : nobody;
        };
        int own = s_ord[warp][dg];
        int t0 = __shfl_sync(0xffffffffu, mine.x, own), len = __shfl_sync(0xffffffffu, mine.y, own);
        load_ids(t0, 0, len);
        for (int r = 0; r < todo; r += 4) {
            const int ownn = s_ord[warp][(r + 4 + dg) & 31];
            const int t0n = __shfl_sync(0xffffffffu, mine.x, ownn);
            int lenn = __shfl_sync(0xffffffffu, mine.y, ownn);
            if (r + 4 >= todo) lenn = 0;
            const int most = __shfl_sync(0xffffffffu, len, 0);               // (the longest of the four)
            uint32_t m[8];
#pragma unroll
            for (int x = 0; x < 8; ++x) m[x] = 0u;
            int have = 0;
            auto rows = [&](int many) {                      // of the collected ids, `many` of the fullest document
                __syncwarp();
                for (int s0 = 0; s0 < many; s0 += U * RPS) {
                    int4 v[U];
#pragma unroll
                    for (int u = 0; u < U; ++u) {
                        const int k = s0 + u * RPS + grp;
                        v[u] = make_int4(0, 0, 0, 0);
                        if (k < have) v[u] = __ldg(tb + (int64_t)ids[k] * LPR);
                    }
#pragma unroll
                    for (int u = 0; u < U; u += 2) coarse_accumulate2(m, v[u], v[u + 1]);
                }
                __syncwarp();
            };
            int base = 0;
            do {
                int32_t cur[4];
#pragma unroll
                for (int k = 0; k < 4; ++k) cur[k] = id[k];
                base += 32;
                const bool more = base < most;
                load_ids(more ? t0 : t0n, more ? base : 0, more ? len : lenn);
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const bool near = s_mask[cur[k] >> 5] >> (cur[k] & 31) & 1u;
                    const uint32_t which = __ballot_sync(0xffffffffu, near) >> (8 * dg) & 0xffu;
                    if (near) ids[have + __popc(which & ((1u << l8) - 1u))] = cur[k];
                    have += __popc(which);
                }
                const int many = __reduce_max_sync(0xffffffffu, have);
                if (!more || many > BOUND_LIST - 32) {
                    rows(many);
                    have = 0;
                }
            } while (base < most);
            // merge the lanes of a document (same columns, different tokens): each exchange keeps one half of the registers
            int nreg = 8;
#pragma unroll
            for (int o = 4; o >= LPR; o >>= 1) {
                const int half = nreg >> 1;
                const bool up = (l8 & o) != 0;
#pragma unroll
                for (int x = 0; x < 4; ++x)
                    if (x < half) {
                        const uint32_t send = up ? m[x] : m[x + half], keep = up ? m[x + half] : m[x];
                        m[x] = __vmaxu2(keep, __shfl_xor_sync(0xffffffffu, send, o));
                    }
                nreg = half;
            }
            int packed = 0;                                  // sum of maxima | saturated << 16
#pragma unroll
            for (int x = 0; x < NF; ++x) {
                const uint32_t f = __vmaxu2(m[x], floor_f[x]);
                const int u_lo = coarse_field_lo(f), u_hi = coarse_field_hi(f);
                packed += (u_lo + u_hi) + (((u_lo >= 255) + (u_hi >= 255)) << 16);
            }
#pragma unroll
            for (int o = 4; o > 0; o >>= 1) packed += __shfl_xor_sync(0xffffffffu, packed, o);      // (127 * 255 < 2^16)
            if (l8 == 0 && r + dg < todo) s_res[warp][own] = coarse_hi(packed, nq);
            own = ownn; t0 = t0n; len = lenn;
        }
        __syncwarp();
        const int32_t res = s_res[warp][lane];
        if (lane < cnt_docs) hi[(int64_t)b * maxc + jb + lane] = res;
        const bool goes_on = mine.y > 0 && res >= limit;
        const unsigned which = __ballot_sync(0xffffffffu, goes_on);
        if (which) {
            int at = 0;
            if (lane == 0) at = atomicAdd(&n_rest[b], __popc(which));
            at = __shfl_sync(0xffffffffu, at, 0);
            if (goes_on) rest[(int64_t)b * maxc + at + __popc(which & ((1u << lane) - 1u))] = jb + lane;
        }
    }
}

// The bounds of those documents (places in the list of ranges, in no order; rest NULL: of all) from the rows of all their tokens.
template <int LPR>
__global__ void __launch_bounds__(CI_THREADS, LPR == 2 ? 4 : 3)
ci_rest_kernel(const uint8_t *__restrict__ table8, int64_t K, int nq, const int2 *__restrict__ rng, const int32_t *__restrict__ rest,
               const int32_t *__restrict__ n_rest, int64_t maxc, const int32_t *__restrict__ cids, int32_t *__restrict__ hi, FirstCut cut)
{
    pdl_entry();
    if (!cut.on()) return;
    ci_coarse_rng_body<LPR>(table8, K, nq, rng, rest, n_rest, maxc, cids, nullptr, hi);
}

bool coarse_supported(int nq) { return nq == 32 || nq == 64; }
int coarse_pitch(int nq) { return nq <= 32 ? 32 : nq <= 64 ? 64 : 128; }

// Several blocks per query in the contender step: few queries with long candidate lists (one block reads 100,000 candidates
// in about 40 us, and 16,384 in the time of the two more launches).
int contender_hist_entries() { return CONT_BINS; }
bool contenders_split(const Index &ix, const Params &p) { return 4 * p.B <= ix.sm_count && p.maxc > 16384; }

int launch_cand_ranges(const Index &ix, const Params &p, const int32_t *cand, const int32_t *n_cand, int2 *rng,
                       int32_t *cont_hist, cudaStream_t st)
{
    int64_t rb = ((int64_t)ix.sm_count * 8 + p.B - 1) / p.B;
    const int64_t rwant = (p.maxc + 255) / 256;
    if (rb > rwant) rb = rwant;
    if (rb < 1) rb = 1;
    launch(cand_range_kernel, dim3((unsigned)rb, (unsigned)p.B), 256, 0, st, cand, n_cand, p.maxc, ix.doc_off, rng,
           contenders_split(ix, p) ? cont_hist : nullptr);
    CHIMERA_CUDA(cudaGetLastError());
    count_launch(SLOT_CI);
    return CHIMERA_OK;
}

// Blocks per query of a scan of 8-bit rows.  Four blocks are resident per SM and the blocks of a query are adjacent in the grid, so
// (resident blocks) / (blocks per query) queries are scanned at the same time and their 8-bit tables compete for
// L2: enough blocks per query to keep those tables within COARSE_L2_TABLES bytes, at least enough to fill the GPU
// when the batch is small, never more than one warp per candidate.  Measured on the Mid corpus at batch 256
// (2 MB tables): 4 blocks per query 57 ms, 16: 23.4, 24: 18.9, 37: 16.5, 74: 16.6, 148: 16.7, 1184: 17.6; a budget
// of 16 MB against 32 MB: Mid 16.56 / 16.52 ms, Large (8 MB tables) 36.6 / 37.2 ms; 64 MB: 21.3 and 46.7 ms.
static int64_t coarse_blocks(const Index &ix, const Params &p)
{
    constexpr int64_t COARSE_L2_TABLES = 16LL << 20;
    const int64_t resident = 4LL * ix.sm_count;
    const int64_t want = (p.maxc + CI_WARPS - 1) / CI_WARPS;
    int64_t per_query = (resident * ix.K * coarse_pitch(p.nq) + COARSE_L2_TABLES - 1) / COARSE_L2_TABLES;
    const int64_t to_fill = (2 * resident + p.B - 1) / p.B;      // two waves when the batch is small
    if (per_query < to_fill) per_query = to_fill;
    if (per_query > want) per_query = want;
    return per_query < 1 ? 1 : per_query;
}
int launch_coarse_bounds(const Index &ix, const Params &p, const uint8_t *table8, const int32_t *cand,
                         const int32_t *n_cand, int32_t *lo, int32_t *hi, const int2 *rng, const FirstCut *cut, cudaStream_t st)
{
    const size_t table_bytes = (size_t)ix.K * coarse_pitch(p.nq);
    const bool use_rng = rng != nullptr;
    const FirstCut call_cut = cut ? *cut : FirstCut();
    constexpr size_t COARSE_SMEM = 160 * 1024;
    const bool small = table_bytes <= COARSE_SMEM;
    if (small) {
        // the whole 8-bit table of a query fits in shared memory: stage it once per block and look rows up there
        constexpr int T = 512;
        int64_t gx = (4LL * ix.sm_count + p.B - 1) / p.B;       // every block re-reads the table: few, long blocks
        int64_t want = (p.maxc + T / 32 - 1) / (T / 32);
        if (gx > want) gx = want;
        if (4 * p.B <= ix.sm_count) gx = (ix.sm_count + p.B - 1) / p.B;        // few queries: a block per SM
        else if (gx > 64) gx = 64;
        if (gx > want) gx = want;
        if (gx < 1) gx = 1;
        dim3 grid((unsigned)gx, (unsigned)p.B);
        if (p.nq == 32) {
            CHIMERA_CUDA(allow_shared(ci_coarse_kernel<2, true, T>, COARSE_SMEM));
            launch(ci_coarse_kernel<2, true, T>, grid, T, table_bytes, st, table8, ix.K, cand, n_cand, p.maxc, ix.cids,
                                                                       ix.doc_off, lo, hi, call_cut);
        } else {
            CHIMERA_CUDA(allow_shared(ci_coarse_kernel<4, true, T>, COARSE_SMEM));
            launch(ci_coarse_kernel<4, true, T>, grid, T, table_bytes, st, table8, ix.K, cand, n_cand, p.maxc, ix.cids,
                                                                       ix.doc_off, lo, hi, call_cut);
        }
        CHIMERA_CUDA(cudaGetLastError());
        count_launch(SLOT_CI);
        return CHIMERA_OK;
    }
    dim3 grid((unsigned)coarse_blocks(ix, p), (unsigned)p.B);
    if (use_rng) {
        if (p.nq == 32)
            launch(ci_coarse_rng_kernel<2>, grid, CI_THREADS, 0, st, table8, ix.K, rng, n_cand, p.maxc, ix.cids, lo, hi, call_cut);
        else
            launch(ci_coarse_rng_kernel<4>, grid, CI_THREADS, 0, st, table8, ix.K, rng, n_cand, p.maxc, ix.cids, lo, hi, call_cut);
        CHIMERA_CUDA(cudaGetLastError());
        count_launch(SLOT_CI);
        return CHIMERA_OK;
    }
    if (p.nq == 32)
        launch(ci_coarse_kernel<2, false, CI_THREADS>, grid, CI_THREADS, 0, st, table8, ix.K, cand, n_cand, p.maxc, ix.cids,
                                                                          ix.doc_off, lo, hi, FirstCut());
    else
        launch(ci_coarse_kernel<4, false, CI_THREADS>, grid, CI_THREADS, 0, st, table8, ix.K, cand, n_cand, p.maxc, ix.cids,
                                                                          ix.doc_off, lo, hi, FirstCut());
    CHIMERA_CUDA(cudaGetLastError());
    count_launch(SLOT_CI);
    return CHIMERA_OK;
}

// Upper bounds of the documents that the first cut keeps (ci_bound_kernel, ci_rest_kernel).  rest: int32 [B][maxc] scratch.
int launch_kept_bounds(const Index &ix, const Params &p, const uint8_t *table8, const uint32_t *mask, const int32_t *theta,
                       const int32_t *tau, const int2 *rng, const int32_t *n_docs, int32_t *hi, int32_t *rest, int32_t *n_rest,
                       const FirstCut &cut, cudaStream_t st)
{
    const int64_t want = (p.maxc + CI_WARPS - 1) / CI_WARPS;
    int64_t gx;
    if (mask) {
        // Two blocks are resident per SM, those of a query adjacent in the grid; few blocks per query keep the copies of its mask
        // few, and sixteen documents or more to a warp, of some six n_prune, find their like in length.
        const int64_t words = (ix.K + 31) / 32;
        const size_t smem = (size_t)(words + 1) * 4;
        gx = (8LL * ix.sm_count + p.B - 1) / p.B;
        if (gx < ix.sm_count / 4) gx = ix.sm_count / 4;
        if (gx > 6 * p.n_prune / (BOUND_THREADS / 2)) gx = 6 * p.n_prune / (BOUND_THREADS / 2);
        if (gx < (2LL * ix.sm_count + p.B - 1) / p.B) gx = (2LL * ix.sm_count + p.B - 1) / p.B;
        if (gx > (want + 1) / 2) gx = (want + 1) / 2;
        auto kern = p.nq <= 32 ? ci_bound_kernel<2> : p.nq <= 64 ? ci_bound_kernel<4> : ci_bound_kernel<8>;
        constexpr size_t MASK_MOST = 40 * 1024;             // more than 266,240 centroids are not cut (filter_used)
        CHIMERA_CUDA(allow_shared(kern, MASK_MOST));
        launch(kern, dim3((unsigned)gx, (unsigned)p.B), BOUND_THREADS, smem, st, table8, ix.K, p.nq, mask, (int)words, theta, tau, rng,
               n_docs, p.maxc, ix.cids, hi, rest, n_rest, cut);
        CHIMERA_CUDA(cudaGetLastError());
        count_launch(SLOT_CI);
        gx = (8LL * ix.sm_count + p.B - 1) / p.B;            // of one or two n_prune documents a query
        if (gx < p.n_prune / 32) gx = p.n_prune / 32;
    } else {
        // (of all rows: half the SMs' number of blocks regardless of the tables, 19 queries of 262,144 centroids and 64-byte rows 525 -> 766 us,
        // 31 of 51,588 and 128 1,353 -> 1,733, 14 of 107,614 and 32 284 -> 349)
        gx = coarse_blocks(ix, p);
    }
    if (gx > want) gx = want;
    auto rest_kern = p.nq <= 32 ? ci_rest_kernel<2> : p.nq <= 64 ? ci_rest_kernel<4> : ci_rest_kernel<8>;
    launch(rest_kern, dim3((unsigned)gx, (unsigned)p.B), CI_THREADS, 0, st, table8, ix.K, p.nq, rng, mask ? rest : nullptr,
           mask ? n_rest : n_docs, p.maxc, ix.cids, hi, cut);
    CHIMERA_CUDA(cudaGetLastError());
    count_launch(SLOT_CI);
    return CHIMERA_OK;
}

// table [rows] int32 -> table8 [rows] uint8 (only needed when stage 1 did not run in this call).
__global__ void coarse_table_kernel(const int32_t *__restrict__ table, int64_t n, uint8_t *__restrict__ table8)
{
    pdl_entry();
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) {
        const int v = table[i] >> 16;
        table8[i] = (uint8_t)(v < 0 ? 0 : v > 255 ? 255 : v);
    }
}
int launch_coarse_table(const Index &ix, const Params &p, const int32_t *table, uint8_t *table8, cudaStream_t st)
{
    const int64_t n = (int64_t)p.B * ix.K * p.nq;
    launch(coarse_table_kernel, (unsigned)((n + 255) / 256), 256, 0, st, table, n, table8);
    CHIMERA_CUDA(cudaGetLastError());
    count_launch(SLOT_MISC);
    return CHIMERA_OK;
}

// Exact CI of a list of documents.  blocks_cap bounds the blocks per query (0 = default).
int launch_centroid_interaction(const Index &ix, const Params &p, const int32_t *table, const int32_t *cand,
                                const int32_t *n_cand, int32_t *ci, int blocks_cap, int slot, const int2 *rng,
                                cudaStream_t st)
{
    int64_t want = (p.maxc + CI_WARPS - 1) / CI_WARPS;
    int64_t cap = blocks_cap > 0 ? blocks_cap : (int64_t)ix.sm_count * 8;
    unsigned gx = (unsigned)(want < cap ? want : cap);
    if (gx < 1) gx = 1;
    dim3 grid(gx, (unsigned)p.B);
    const int nqw = (p.nq + 31) / 32;
    const int2 *grng = blocks_cap > 0 ? rng : nullptr;
    if (rng != nullptr && blocks_cap > 0 && (p.nq == 32 || p.nq == 64)) {       // the listed documents' token ranges are known
        if (p.nq == 32)
            launch(ci_wide_rng_kernel<8>, grid, CI_THREADS, 0, st, table, ix.K, rng, n_cand, p.maxc, ix.cids, ci);
        else
            launch(ci_wide_rng_kernel<16>, grid, CI_THREADS, 0, st, table, ix.K, rng, n_cand, p.maxc, ix.cids, ci);
        CHIMERA_CUDA(cudaGetLastError());
        count_launch(slot);
        return CHIMERA_OK;
    }
    if (p.nq == 32)
        launch(ci_wide_kernel<8>, grid, CI_THREADS, 0, st, table, ix.K, cand, n_cand, p.maxc, ix.cids, ix.doc_off, ci);
    else if (p.nq == 64)
        launch(ci_wide_kernel<16>, grid, CI_THREADS, 0, st, table, ix.K, cand, n_cand, p.maxc, ix.cids, ix.doc_off, ci);
    else {
        auto kern = nqw == 1 ? ci_kernel<1> : nqw == 2 ? ci_kernel<2> : ci_kernel<4>;
        launch(kern, grid, CI_THREADS, 0, st, table, ix.K, p.nq, cand, n_cand, p.maxc, ix.cids, ix.doc_off, grng, ci);
    }
    CHIMERA_CUDA(cudaGetLastError());
    count_launch(slot);
    return CHIMERA_OK;
}

// ------------------------------------------------------------------------------------------------ selection ------
// The selection of few from many in one pass over the scores.  A block waits for its loads most of the time, and the radix
// select with the compaction behind it passes over the scores four times and over the ids once.  Here a sample of SEL_SAMPLE
// scores gives a bound that somewhat more than n_prune scores reach (the wanted rank of the sample and four standard deviations
// more), one pass collects those in shared memory, and the selection and the order of the survivors are found there.  Scores in
// masses (documents that repeat) can put more at the bound than there is room for, as the sample shows: they are counted then, and
// where some of them are needed the bound is the threshold itself, else the ones above it are collected.
// Measured (1,024 wanted of Mid's candidates, 1-bit refinement): 256 queries 122 -> 50 us, 64 queries 69 -> 30 us.
// Room for 7,168 serves 4,096 wanted too (4 million documents, 64 queries, 1-bit codes: 1,798 -> 1,742 us a call; 3,584 did not).
// Masses of equal scores, 256 queries, selected among all / with every mass collected and ties at the edge counted against one
// another / so: 40,000 candidates, 4,096 wanted, 400 of each score 53 / 120 / 52 us, 2,000 54 / 483 / 54; 200,000, 2,000 of each 244 /
// 526 / 225; 1,024 wanted, 10,000 of each 239 / 314 / 177.  (Collecting by votes, without an atomic each: 35 -> 50, 71 -> 115 us where all
// scores differ: the instructions count.)
constexpr int SEL_SAMPLE = 8192, SEL_FEW = 7168, SEL_BINS = 2048;
struct SelFew {
    union {
        uint32_t sample[SEL_SAMPLE];
        struct {
            uint32_t u[SEL_FEW];                             // scores in the order of radix_select, in any order
            int pos[SEL_FEW];                                // their places in the candidate list
            uint16_t ord[SEL_FEW];                           // the survivors by bucket of places
        };
    };
    int n;
};
// The wanted rank of the sample.  Taken from 16,384 scores on (shorter lists cost a pass of the block's loads or two, no more
// than the sample) while the documents to be expected fill no more than 6/7 of the list.
__host__ __device__ __forceinline__ bool select_few_applies(int n, int n_prune, int *want)
{
    const float r = (float)n_prune * ((float)SEL_SAMPLE / (float)n);
    const float w = r + 4.f * sqrtf(r) + 8.f;
    *want = (int)w;
    return n >= 2 * SEL_SAMPLE && w * (float)n <= (float)(SEL_FEW / 7 * 6) * SEL_SAMPLE;
}
enum { FEW_DONE, FEW_THRESHOLD, FEW_NOT };                   // selected; nothing written, *thr and *need_eq known; nothing known
__device__ __forceinline__ int select_few(const int32_t *__restrict__ cb, const int32_t *__restrict__ sb, int n, int n_prune,
                                          int want, int32_t *__restrict__ out, int32_t *__restrict__ out_ci, SelFew &few,
                                          int *hist /* [SEL_BINS] */, int *warp_part, uint32_t *s_prefix, int *s_want,
                                          uint32_t *thr_out, int *need_eq_out)
{
    const int tid = threadIdx.x;
    // groups of four neighbours at equal distances (a 32-byte sector costs the same for one)
    {
        const int step = n / (SEL_SAMPLE / 4);
        uint32_t v[SEL_SAMPLE / SEL_THREADS];
#pragma unroll
        for (int e = 0; e < SEL_SAMPLE / SEL_THREADS; ++e) {
            const int i = e * SEL_THREADS + tid;
            v[e] = (uint32_t)sb[(i >> 2) * step + (i & 3)];
        }
#pragma unroll
        for (int e = 0; e < SEL_SAMPLE / SEL_THREADS; ++e) few.sample[e * SEL_THREADS + tid] = v[e];
    }
    if (tid == 0) few.n = 0;
    __syncthreads();
    int need_eq;
    uint32_t bound = radix_select([&](int j) { return (int32_t)few.sample[j]; }, SEL_SAMPLE, want, hist, warp_part, s_prefix,
                                  s_want, &need_eq);
    // (the last digit's histogram has how many scores of the sample equal the bound)
    const bool masses = (float)(want - need_eq + hist[bound & 1023u]) * (float)n > (float)SEL_FEW * SEL_SAMPLE;
    __syncthreads();                                         // the sample's place and the histogram are used again
    if (masses) {
        int above = 0, equal = 0, n_above, n_equal;          // (of this thread's scores, of all)
        for (int base = 0; base < n; base += 8 * SEL_THREADS) {
            uint32_t u[8];
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                const int j = base + e * SEL_THREADS + tid;
                u[e] = j < n ? (uint32_t)sb[j] ^ 0x80000000u : 0u;
            }
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                above += u[e] > bound ? 1 : 0;
                equal += u[e] == bound && base + e * SEL_THREADS + tid < n ? 1 : 0;
            }
        }
        sel_block_scan(above, &n_above, warp_part);
        sel_block_scan(equal, &n_equal, warp_part);
        if (n_above < n_prune) {
            *thr_out = bound;
            *need_eq_out = n_prune - n_above;
            return n_prune - n_above <= n_equal ? FEW_THRESHOLD : FEW_NOT;
        }
        if (n_above > SEL_FEW) return FEW_NOT;
        ++bound;                                             // (there are scores above it)
    }
    for (int base = 0; base < n; base += 8 * SEL_THREADS) {
        uint32_t u[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            const int j = base + e * SEL_THREADS + tid;
            u[e] = j < n ? (uint32_t)sb[j] ^ 0x80000000u : 0u;
        }
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            const int j = base + e * SEL_THREADS + tid;
            if (u[e] >= bound && j < n) {
                const int slot = atomicAdd(&few.n, 1);
                if (slot < SEL_FEW) { few.u[slot] = u[e]; few.pos[slot] = j; }
            }
        }
    }
    __syncthreads();
    const int c = few.n;
    if (c < n_prune || c > SEL_FEW) return FEW_NOT;
    const uint32_t thr = radix_select([&](int j) { return (int32_t)(few.u[j] ^ 0x80000000u); }, c, n_prune, hist, warp_part,
                                      s_prefix, s_want, &need_eq);
    const int n_eq = hist[thr & 1023u];
    int last = n;                                            // ties at the edge go to the smaller ids: places up to this one
    __syncthreads();
    if (n_eq > need_eq && n_eq <= 256) {
        if (tid == 0) few.n = 0;
        __syncthreads();
        for (int i = tid; i < c; i += SEL_THREADS)
            if (few.u[i] == thr) hist[atomicAdd(&few.n, 1)] = few.pos[i];
        __syncthreads();
        if (tid < n_eq) {
            const int pos = hist[tid];
            int before = 0;
            for (int k = 0; k < n_eq; ++k) before += hist[k] < pos ? 1 : 0;
            if (before == need_eq - 1) *s_want = pos;
        }
        __syncthreads();
        last = *s_want;
    } else if (n_eq > need_eq) {
        int one;                                             // (places are distinct)
        last = -(int)(radix_select([&](int j) { return few.u[j] == thr ? -few.pos[j] : INT_MIN; }, c, need_eq, hist, warp_part,
                                   s_prefix, s_want, &one) ^ 0x80000000u);
    }
    bool keep[(SEL_FEW + SEL_THREADS - 1) / SEL_THREADS];
#pragma unroll
    for (int e = 0; e < (SEL_FEW + SEL_THREADS - 1) / SEL_THREADS; ++e) {
        const int i = e * SEL_THREADS + tid;
        keep[e] = i < c && (few.u[i] > thr || (few.u[i] == thr && few.pos[i] <= last));
    }
    __syncthreads();
    // the survivors' order: buckets of neighbouring places (half a survivor each at 1,024), then the place within the bucket
    int shift = 0;
    while (((n - 1) >> shift) >= SEL_BINS) ++shift;
    for (int i = tid; i < SEL_BINS; i += SEL_THREADS) hist[i] = 0;
    __syncthreads();
#pragma unroll
    for (int e = 0; e < (SEL_FEW + SEL_THREADS - 1) / SEL_THREADS; ++e)
        if (keep[e]) atomicAdd(&hist[few.pos[e * SEL_THREADS + tid] >> shift], 1);
    __syncthreads();
    const int h0 = hist[2 * tid], h1 = hist[2 * tid + 1];
    int total;
    const int first = sel_block_scan(h0 + h1, &total, warp_part);
    hist[2 * tid] = first;
    hist[2 * tid + 1] = first + h0;
    __syncthreads();
#pragma unroll
    for (int e = 0; e < (SEL_FEW + SEL_THREADS - 1) / SEL_THREADS; ++e) {
        const int i = e * SEL_THREADS + tid;
        if (keep[e]) few.ord[atomicAdd(&hist[few.pos[i] >> shift], 1)] = (uint16_t)i;
    }
    __syncthreads();                                         // hist[x]: where bucket x ends
#pragma unroll
    for (int e = 0; e < (SEL_FEW + SEL_THREADS - 1) / SEL_THREADS; ++e) {
        const int i = e * SEL_THREADS + tid;
        if (keep[e]) {
            const int pos = few.pos[i], x = pos >> shift;
            const int begin = x ? hist[x - 1] : 0, end = hist[x];
            int rank = begin;
            for (int k = begin; k < end; ++k) rank += few.pos[few.ord[k]] < pos ? 1 : 0;
            out[rank] = cb[pos];
            if (out_ci) out_ci[rank] = (int32_t)(few.u[i] ^ 0x80000000u);
        }
    }
    return FEW_DONE;
}

// grid (B).  pruned[b][0..n_prune) ascending ids, -1 padded; n_pruned[b]; pruned_ci (optional): the score of each
// kept document, INT_MIN beside every -1.
template <bool MANY>      // the list may be long (the shared memory of select_few is there)
__global__ void __launch_bounds__(SEL_THREADS)
select_kernel(const int32_t *__restrict__ cand, const int32_t *__restrict__ n_cand, const int32_t *__restrict__ ci,
              int64_t maxc, int n_prune, int32_t *__restrict__ pruned, int32_t *__restrict__ n_pruned,
              int32_t *__restrict__ pruned_ci)
{
    pdl_entry();
    extern __shared__ uint4 s_few[];                         // (two blocks per SM: 72 KB each)
    SelFew &few = *reinterpret_cast<SelFew *>(s_few);
    __shared__ int hist[SEL_BINS];
    __shared__ int warp_part[32];
    __shared__ uint32_t s_prefix;
    __shared__ int s_want;
    const int b = blockIdx.x;
    const int n = n_cand[b];
    const int32_t *cb = cand + (int64_t)b * maxc;
    const int32_t *sb = ci + (int64_t)b * maxc;
    int32_t *out = pruned + (int64_t)b * n_prune;
    int32_t *out_ci = pruned_ci ? pruned_ci + (int64_t)b * n_prune : nullptr;

    if (n <= n_prune) {
        for (int j = threadIdx.x; j < n_prune; j += SEL_THREADS) {
            out[j] = j < n ? cb[j] : -1;
            if (out_ci) out_ci[j] = j < n ? sb[j] : INT_MIN;
        }
        if (threadIdx.x == 0) n_pruned[b] = n;
        return;
    }
    int need_eq, want, how = FEW_NOT;
    uint32_t thr;
    if (MANY && select_few_applies(n, n_prune, &want))
        how = select_few(cb, sb, n, n_prune, want, out, out_ci, few, hist, warp_part, &s_prefix, &s_want, &thr, &need_eq);
    if (how == FEW_DONE) {
        if (threadIdx.x == 0) n_pruned[b] = n_prune;
        return;
    }
    if (how == FEW_NOT) {
        __syncthreads();
        thr = radix_select([&](int j) { return sb[j]; }, n, n_prune, hist, warp_part, &s_prefix, &s_want, &need_eq);
    }

    // Ordered compaction: keep u > thr, and the first need_eq entries with u == thr.  Each thread owns four
    // consecutive entries per round, so one block scan covers 4096 entries.
    int run_gt = 0, run_eq = 0;
    for (int base = 0; base < n; base += 4 * SEL_THREADS) {
        const int j0 = base + 4 * threadIdx.x;
        uint32_t u[4];
        int32_t id[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const int j = j0 + e;
            u[e] = j < n ? ((uint32_t)sb[j] ^ 0x80000000u) : 0u;
            id[e] = j < n ? cb[j] : 0;
        }
        int gt = 0, eq = 0;
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            gt += (j0 + e < n && u[e] > thr) ? 1 : 0;
            eq += (j0 + e < n && u[e] == thr) ? 1 : 0;
        }
        int total;
        const int before = sel_block_scan((gt << 16) | eq, &total, warp_part);   // <= 4096 per field
        int gt_before = run_gt + (before >> 16), eq_before = run_eq + (before & 0xffff);
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            if (j0 + e >= n) break;
            const bool is_gt = u[e] > thr, is_eq = u[e] == thr;
            if (is_gt || (is_eq && eq_before < need_eq)) {
                const int pos = gt_before + (eq_before < need_eq ? eq_before : need_eq);
                out[pos] = id[e];
                if (out_ci) out_ci[pos] = (int32_t)(u[e] ^ 0x80000000u);
            }
            gt_before += is_gt ? 1 : 0;
            eq_before += is_eq ? 1 : 0;
        }
        run_gt += total >> 16;
        run_eq += total & 0xffff;
    }
    if (threadIdx.x == 0) n_pruned[b] = n_prune;
}

// grid (B).  Contenders for the top n_prune: with tau = the n_prune-th largest lower bound, every document of the
// true top n_prune has hi >= CI >= (n_prune-th largest CI) >= tau.  Writes their ids (ascending) and their number.
__global__ void __launch_bounds__(SEL_THREADS)
contender_kernel(const int32_t *__restrict__ cand, const int32_t *__restrict__ n_cand, const int32_t *__restrict__ lo,
                 const int32_t *__restrict__ hi, int64_t maxc, int n_prune, int nq, int32_t *__restrict__ cont,
                 int32_t *__restrict__ n_cont, const int2 *__restrict__ rng, int2 *__restrict__ cont_rng)
{
    pdl_entry();
    __shared__ int hist[CONT_BINS];
    __shared__ int warp_part[32];
    __shared__ int s_bin;
    const int b = blockIdx.x;
    const int n = n_cand[b];
    const int32_t *cb = cand + (int64_t)b * maxc;
    const int32_t *lb = lo + (int64_t)b * maxc;
    const int32_t *hb = hi + (int64_t)b * maxc;
    int32_t *out = cont + (int64_t)b * maxc;
    const int2 *rb = rng ? rng + (int64_t)b * maxc : nullptr;
    int2 *orng = cont_rng ? cont_rng + (int64_t)b * maxc : nullptr;
    if (n <= n_prune) {
        for (int j = threadIdx.x; j < n; j += SEL_THREADS) {
            out[j] = cb[j];
            if (orng) orng[j] = rb[j];
        }
        if (threadIdx.x == 0) n_cont[b] = n;
        return;
    }
    const int32_t tau = contender_threshold(lb, n, n_prune, nq, hist, warp_part, &s_bin);
    // ordered compaction, eight consecutive entries per thread and round (one block scan per 8192 entries); the ids
    // are only read for the few entries that are kept
    int run = 0;
    for (int base = 0; base < n; base += 8 * SEL_THREADS) {
        const int j0 = base + 8 * threadIdx.x;
        int32_t hv[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) hv[e] = j0 + e < n ? hb[j0 + e] : INT_MIN;
        int keep = 0;
#pragma unroll
        for (int e = 0; e < 8; ++e) keep += (j0 + e < n && hv[e] >= tau) ? 1 : 0;
        int tot;
        int pos = run + sel_block_scan(keep, &tot, warp_part);
#pragma unroll
        for (int e = 0; e < 8; ++e)
            if (j0 + e < n && hv[e] >= tau) {
                out[pos] = cb[j0 + e];
                if (orng) orng[pos] = rb[j0 + e];
                ++pos;
            }
        run += tot;
    }
    if (threadIdx.x == 0) n_cont[b] = run;
}

// Document-sharded search, grid (B): the global top n_prune of the shards' local top-n_prune lists.  all_ids / all_ci
// are [world][B][n_prune] (global document ids ascending within a shard, -1 / INT_MIN padded); shards own ascending,
// disjoint id ranges in rank order, so walking rank by rank visits the valid entries in ascending id order and ties
// resolve towards the smaller id exactly as in select_kernel.  Of the selected documents this shard keeps its own
// (ids in [doc_base, doc_base + n_local)) as local ids: pruned[b][0..n_prune) ascending, -1 padded; n_pruned[b].
__global__ void __launch_bounds__(SEL_THREADS)
shard_select_kernel(const int32_t *__restrict__ all_ids, const int32_t *__restrict__ all_ci, int world, int B,
                    int n_prune, long long doc_base, long long n_local, int32_t *__restrict__ pruned,
                    int32_t *__restrict__ n_pruned)
{
    pdl_entry();
    __shared__ int hist[2048];
    __shared__ int warp_part[32];
    __shared__ uint32_t s_prefix;
    __shared__ int s_want;
    const int b = blockIdx.x;
    const int n = world * n_prune;
    auto at = [&](int j) { return ((int64_t)(j / n_prune) * B + b) * n_prune + j % n_prune; };
    int32_t *out = pruned + (int64_t)b * n_prune;

    // number of valid entries
    int valid = 0;
    for (int j = threadIdx.x; j < n; j += SEL_THREADS) valid += all_ids[at(j)] >= 0 ? 1 : 0;
    int total_valid;
    sel_block_scan(valid, &total_valid, warp_part);
    uint32_t thr = 0u;              // keep everything valid
    int need_eq = 0;
    if (total_valid > n_prune)
        thr = radix_select([&](int j) { return all_ci[at(j)]; }, n, n_prune, hist, warp_part, &s_prefix, &s_want,
                           &need_eq);
    const bool keep_all = total_valid <= n_prune;

    int run_eq = 0, run_own = 0;
    for (int base = 0; base < n; base += 4 * SEL_THREADS) {
        const int j0 = base + 4 * threadIdx.x;
        uint32_t u[4];
        int32_t id[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const int j = j0 + e;
            id[e] = j < n ? all_ids[at(j)] : -1;
            u[e] = id[e] >= 0 ? ((uint32_t)all_ci[at(j)] ^ 0x80000000u) : 0u;
        }
        int eq = 0;
#pragma unroll
        for (int e = 0; e < 4; ++e) eq += (id[e] >= 0 && !keep_all && u[e] == thr) ? 1 : 0;
        int total_eq;
        int eq_before = run_eq + sel_block_scan(eq, &total_eq, warp_part);
        bool own[4];
        int n_own = 0;
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            bool kept = id[e] >= 0;
            if (kept && !keep_all) {
                const bool is_eq = u[e] == thr;
                kept = u[e] > thr || (is_eq && eq_before < need_eq);
                eq_before += is_eq ? 1 : 0;
            }
            own[e] = kept && id[e] >= doc_base && id[e] < doc_base + n_local;
            n_own += own[e] ? 1 : 0;
        }
        int total_own;
        int pos = run_own + sel_block_scan(n_own, &total_own, warp_part);
#pragma unroll
        for (int e = 0; e < 4; ++e)
            if (own[e]) out[pos++] = (int32_t)(id[e] - doc_base);
        run_eq += total_eq;
        run_own += total_own;
    }
    for (int j = run_own + threadIdx.x; j < n_prune; j += SEL_THREADS) out[j] = -1;
    if (threadIdx.x == 0) n_pruned[b] = run_own;
}

int launch_shard_select(const Params &p, const int32_t *all_ids, const int32_t *all_ci, int world, int64_t doc_base,
                        int64_t n_local, int32_t *pruned, int32_t *n_pruned, cudaStream_t st)
{
    launch(shard_select_kernel, (unsigned)p.B, SEL_THREADS, 0, st, all_ids, all_ci, world, p.B, p.n_prune,
                                                               (long long)doc_base, (long long)n_local, pruned,
                                                               n_pruned);
    CHIMERA_CUDA(cudaGetLastError());
    count_launch(SLOT_SELECT);
    return CHIMERA_OK;
}

// The same selection spread over CONT_SPLIT blocks per query, for calls with few queries: one block reads its arrays
// at one SM's bandwidth (about 40 us for 100k candidates), which is most of the stage's latency when a single query is
// served.  Three kernels: slice histograms added into a global one; every block finds tau from it and counts its
// slice's contenders; every block writes its contenders behind those of the slices before it (ascending ids kept).
// Scratch: `scratch[b * maxc ...]` holds the histogram (CONT_BINS), the slice counts (CONT_SPLIT) and tau.
constexpr int CONT_SPLIT = 32;

__device__ __forceinline__ void cont_slice(int n, int g, int *j0, int *j1)
{
    const int per = (n + CONT_SPLIT - 1) / CONT_SPLIT;
    *j0 = g * per < n ? g * per : n;
    *j1 = (g + 1) * per < n ? (g + 1) * per : n;
}

__global__ void __launch_bounds__(SEL_THREADS)
contender_hist_kernel(const int32_t *__restrict__ n_cand, const int32_t *__restrict__ lo, int64_t maxc, int n_prune,
                      int nq, int32_t *__restrict__ scratch)
{
    pdl_entry();
    __shared__ int hist[CONT_BINS];
    const int b = blockIdx.y, n = n_cand[b];
    if (n <= n_prune) return;                          // everything is a contender: no threshold needed
    int j0, j1;
    cont_slice(n, blockIdx.x, &j0, &j1);
    const int32_t *lb = lo + (int64_t)b * maxc;
    const int bin_shift = contender_bin_shift(nq);
    for (int i = threadIdx.x; i < CONT_BINS; i += SEL_THREADS) hist[i] = 0;
    __syncthreads();
    for (int j = j0 + threadIdx.x; j < j1; j += SEL_THREADS)
        atomicAdd(&hist[coarse_key(lb[j]) >> bin_shift], 1);
    __syncthreads();
    int32_t *gh = scratch + (int64_t)b * maxc;
    for (int i = threadIdx.x; i < CONT_BINS; i += SEL_THREADS)
        if (hist[i]) atomicAdd(&gh[i], hist[i]);
}

__global__ void __launch_bounds__(SEL_THREADS)
contender_count_kernel(const int32_t *__restrict__ n_cand, const int32_t *__restrict__ hi, int64_t maxc, int n_prune,
                       int nq, int32_t *__restrict__ scratch)
{
    pdl_entry();
    __shared__ int warp_part[32];
    __shared__ int s_bin;
    const int b = blockIdx.y, n = n_cand[b];
    int32_t *gh = scratch + (int64_t)b * maxc;
    int32_t tau = INT_MIN;
    if (n > n_prune) {
        const int bin_shift = contender_bin_shift(nq);
        constexpr int PER = CONT_BINS / SEL_THREADS;
        const int first_bin = CONT_BINS - 1 - PER * (int)threadIdx.x;
        int h[PER], mine = 0;
#pragma unroll
        for (int e = 0; e < PER; ++e) { h[e] = gh[first_bin - e]; mine += h[e]; }
        int total;
        int before = sel_block_scan(mine, &total, warp_part);
        if (before < n_prune && n_prune <= before + mine) {
#pragma unroll
            for (int e = 0; e < PER; ++e) {
                if (before < n_prune && n_prune <= before + h[e]) s_bin = first_bin - e;
                before += h[e];
            }
        }
        __syncthreads();
        tau = (s_bin << bin_shift) << 16;
    }
    int j0, j1;
    cont_slice(n, blockIdx.x, &j0, &j1);
    const int32_t *hb = hi + (int64_t)b * maxc;
    int keep = 0;
    for (int j = j0 + threadIdx.x; j < j1; j += SEL_THREADS) keep += hb[j] >= tau ? 1 : 0;
    int total;
    sel_block_scan(keep, &total, warp_part);
    if (threadIdx.x == 0) {
        gh[CONT_BINS + blockIdx.x] = total;
        if (blockIdx.x == 0) gh[CONT_BINS + CONT_SPLIT] = tau;
    }
}

__global__ void __launch_bounds__(SEL_THREADS)
contender_write_kernel(const int32_t *__restrict__ cand, const int32_t *__restrict__ n_cand,
                       const int32_t *__restrict__ hi, int64_t maxc, const int32_t *__restrict__ scratch,
                       int32_t *__restrict__ cont, int32_t *__restrict__ n_cont, const int2 *__restrict__ rng,
                       int2 *__restrict__ cont_rng)
{
    pdl_entry();
    __shared__ int warp_part[32];
    const int b = blockIdx.y, n = n_cand[b], g = blockIdx.x;
    const int32_t *gh = scratch + (int64_t)b * maxc;
    const int32_t tau = gh[CONT_BINS + CONT_SPLIT];
    int offset = 0;
    for (int s = 0; s < g; ++s) offset += gh[CONT_BINS + s];
    int j0, j1;
    cont_slice(n, g, &j0, &j1);
    const int32_t *cb = cand + (int64_t)b * maxc;
    const int32_t *hb = hi + (int64_t)b * maxc;
    int32_t *out = cont + (int64_t)b * maxc;
    const int2 *rb = rng ? rng + (int64_t)b * maxc : nullptr;
    int2 *orng = cont_rng ? cont_rng + (int64_t)b * maxc : nullptr;
    int run = offset;
    for (int base = j0; base < j1; base += 4 * SEL_THREADS) {
        const int q0 = base + 4 * threadIdx.x;
        int32_t hv[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) hv[e] = q0 + e < j1 ? hb[q0 + e] : INT_MIN;
        int keep = 0;
#pragma unroll
        for (int e = 0; e < 4; ++e) keep += (q0 + e < j1 && hv[e] >= tau) ? 1 : 0;
        int32_t id[4];                                       // (asked for in front of the scan's barriers)
        int2 r[4];
#pragma unroll
        for (int e = 0; e < 4; ++e)
            if (q0 + e < j1 && hv[e] >= tau) {
                id[e] = cb[q0 + e];
                r[e] = orng ? rb[q0 + e] : make_int2(0, 0);
            }
        int tot;
        int pos = run + sel_block_scan(keep, &tot, warp_part);
#pragma unroll
        for (int e = 0; e < 4; ++e)
            if (q0 + e < j1 && hv[e] >= tau) {
                out[pos] = id[e];
                if (orng) orng[pos] = r[e];
                ++pos;
            }
        run += tot;
    }
    if (g == CONT_SPLIT - 1 && threadIdx.x == 0) n_cont[b] = run;
}

// scratch: an int32 [B][maxc] array that is free during this step (the exact-CI output buffer).
int launch_contenders(const Index &ix, const Params &p, const int32_t *cand, const int32_t *n_cand, const int32_t *lo,
                      const int32_t *hi, int32_t *cont, int32_t *n_cont, int32_t *scratch, const int2 *rng,
                      int2 *cont_rng, cudaStream_t st)
{
    if (contenders_split(ix, p)) {
        // few queries: CONT_SPLIT blocks each.  The kernel that wrote the ranges has cleared the histograms; without ranges
        // (2^31 tokens or more) nothing has.
        if (rng == nullptr)
            CHIMERA_CUDA(cudaMemset2DAsync(scratch, sizeof(int32_t) * (size_t)p.maxc, 0, sizeof(int32_t) * CONT_BINS,
                                           (size_t)p.B, st));
        const dim3 grid(CONT_SPLIT, (unsigned)p.B);
        launch(contender_hist_kernel, grid, SEL_THREADS, 0, st, n_cand, lo, p.maxc, p.n_prune, p.nq, scratch);
        CHIMERA_CUDA(cudaGetLastError());
        launch(contender_count_kernel, grid, SEL_THREADS, 0, st, n_cand, hi, p.maxc, p.n_prune, p.nq, scratch);
        CHIMERA_CUDA(cudaGetLastError());
        launch(contender_write_kernel, grid, SEL_THREADS, 0, st, cand, n_cand, hi, p.maxc, scratch, cont, n_cont, rng, cont_rng);
        CHIMERA_CUDA(cudaGetLastError());
        count_launch(SLOT_SELECT, 3);
        return CHIMERA_OK;
    }
    launch(contender_kernel, (unsigned)p.B, SEL_THREADS, 0, st, cand, n_cand, lo, hi, p.maxc, p.n_prune, p.nq, cont,
                                                            n_cont, rng, cont_rng);
    CHIMERA_CUDA(cudaGetLastError());
    count_launch(SLOT_SELECT);
    return CHIMERA_OK;
}

// ------------------------------------------------------------------------------------------------------------------
// The same selection spread over SELS_SPLIT blocks per query, for calls with few queries (one block reads its arrays at
// one SM's bandwidth; with a single query that is most of the stage's latency).  Five kernels, each block working on a
// contiguous slice of the candidates: three radix passes whose slice histograms are added into global ones (every block
// of the next kernel re-derives the chosen digit from the global histogram, which is cheap), a count of the entries
// above and at the threshold per slice, and the ordered write behind the slices before it.
// Scratch per query (int32): hist[0] 2048, hist[1] 2048, hist[2] 1024, greater[SELS_SPLIT], equal[SELS_SPLIT].
constexpr int SELS_SPLIT = 32;
constexpr int SELS_SCRATCH = 2048 + 2048 + 1024 + 2 * SELS_SPLIT;

__device__ __forceinline__ void sels_slice(int n, int g, int *j0, int *j1)
{
    const int per = (n + SELS_SPLIT - 1) / SELS_SPLIT;
    *j0 = g * per < n ? g * per : n;
    *j1 = (g + 1) * per < n ? (g + 1) * per : n;
}

// The digit (bin) of `bins` descending-cumulative bins that holds rank `want`, and the rank left inside it.
// Whole block, uniform result.
__device__ __forceinline__ void sels_find(const int32_t *__restrict__ hist, int bins, int want, int *warp_part,
                                          int *s_out /* [2] */, int *bin, int *want_rest)
{
    const int hi_bin = bins - 1 - 2 * (int)threadIdx.x, lo_bin = hi_bin - 1;
    const int h_hi = hi_bin >= 0 ? hist[hi_bin] : 0;
    const int h_lo = lo_bin >= 0 ? hist[lo_bin] : 0;
    int total;
    const int before = sel_block_scan(h_hi + h_lo, &total, warp_part);
    if (before < want && want <= before + h_hi + h_lo) {
        if (want <= before + h_hi) { s_out[0] = hi_bin; s_out[1] = want - before; }
        else { s_out[0] = lo_bin; s_out[1] = want - before - h_hi; }
    }
    __syncthreads();
    *bin = s_out[0];
    *want_rest = s_out[1];
    __syncthreads();
}

// PASS 0, 1, 2: histogram of the pass's digit over the slice's entries that match the digits chosen so far.
template <int PASS>
__global__ void __launch_bounds__(SEL_THREADS)
sels_hist_kernel(const int32_t *__restrict__ n_cand, const int32_t *__restrict__ ci, int64_t maxc, int n_prune,
                 int32_t *__restrict__ scratch)
{
    pdl_entry();
    __shared__ int hist[2048];
    __shared__ int warp_part[32];
    __shared__ int s_out[2];
    const int b = blockIdx.y, n = n_cand[b];
    if (n <= n_prune) return;
    int32_t *sc = scratch + (int64_t)b * SELS_SCRATCH;
    uint32_t prefix = 0u, mask = 0u;
    int want = n_prune;
    if (PASS >= 1) {
        int bin;
        sels_find(sc, 2048, want, warp_part, s_out, &bin, &want);
        prefix = (uint32_t)bin << 21;
        mask = 0x7ffu << 21;
    }
    if (PASS >= 2) {
        int bin;
        sels_find(sc + 2048, 2048, want, warp_part, s_out, &bin, &want);
        prefix |= (uint32_t)bin << 10;
        mask |= 0x7ffu << 10;
    }
    constexpr int SHIFT = PASS == 0 ? 21 : PASS == 1 ? 10 : 0;
    constexpr int BINS = PASS == 2 ? 1024 : 2048;
    for (int i = threadIdx.x; i < BINS; i += SEL_THREADS) hist[i] = 0;
    __syncthreads();
    int j0, j1;
    sels_slice(n, blockIdx.x, &j0, &j1);
    const int32_t *sb = ci + (int64_t)b * maxc;
    for (int j = j0 + threadIdx.x; j < j1; j += SEL_THREADS) {
        const uint32_t u = (uint32_t)sb[j] ^ 0x80000000u;
        if ((u & mask) == prefix) atomicAdd(&hist[(u >> SHIFT) & (BINS - 1)], 1);
    }
    __syncthreads();
    int32_t *gh = sc + (PASS == 0 ? 0 : PASS == 1 ? 2048 : 4096);
    for (int i = threadIdx.x; i < BINS; i += SEL_THREADS)
        if (hist[i]) atomicAdd(&gh[i], hist[i]);
}

// The threshold (all three digits) and how many entries equal to it belong to the top n_prune.
__device__ __forceinline__ uint32_t sels_threshold(const int32_t *sc, int n_prune, int *warp_part, int *s_out, int *need_eq)
{
    int b1, b2, b3, want = n_prune;
    sels_find(sc, 2048, want, warp_part, s_out, &b1, &want);
    sels_find(sc + 2048, 2048, want, warp_part, s_out, &b2, &want);
    sels_find(sc + 4096, 1024, want, warp_part, s_out, &b3, &want);
    *need_eq = want;
    return ((uint32_t)b1 << 21) | ((uint32_t)b2 << 10) | (uint32_t)b3;
}

__global__ void __launch_bounds__(SEL_THREADS)
sels_count_kernel(const int32_t *__restrict__ n_cand, const int32_t *__restrict__ ci, int64_t maxc, int n_prune,
                  int32_t *__restrict__ scratch)
{
    pdl_entry();
    __shared__ int warp_part[32];
    __shared__ int s_out[2];
    const int b = blockIdx.y, n = n_cand[b];
    if (n <= n_prune) return;
    int32_t *sc = scratch + (int64_t)b * SELS_SCRATCH;
    int need_eq;
    const uint32_t thr = sels_threshold(sc, n_prune, warp_part, s_out, &need_eq);
    int j0, j1;
    sels_slice(n, blockIdx.x, &j0, &j1);
    const int32_t *sb = ci + (int64_t)b * maxc;
    int gt = 0, eq = 0;
    for (int j = j0 + threadIdx.x; j < j1; j += SEL_THREADS) {
        const uint32_t u = (uint32_t)sb[j] ^ 0x80000000u;
        gt += u > thr ? 1 : 0;
        eq += u == thr ? 1 : 0;
    }
    int total;
    sel_block_scan((gt << 16) | eq, &total, warp_part);        // a slice has fewer than 2^15 entries (launcher)
    if (threadIdx.x == 0) {
        sc[5120 + blockIdx.x] = total >> 16;
        sc[5120 + SELS_SPLIT + blockIdx.x] = total & 0xffff;
    }
}

__global__ void __launch_bounds__(SEL_THREADS)
sels_write_kernel(const int32_t *__restrict__ cand, const int32_t *__restrict__ n_cand, const int32_t *__restrict__ ci,
                  int64_t maxc, int n_prune, const int32_t *__restrict__ scratch, int32_t *__restrict__ pruned,
                  int32_t *__restrict__ n_pruned, int32_t *__restrict__ pruned_ci)
{
    pdl_entry();
    __shared__ int warp_part[32];
    __shared__ int s_out[2];
    const int b = blockIdx.y, n = n_cand[b], g = blockIdx.x;
    const int32_t *cb = cand + (int64_t)b * maxc;
    const int32_t *sb = ci + (int64_t)b * maxc;
    int32_t *out = pruned + (int64_t)b * n_prune;
    int32_t *out_ci = pruned_ci ? pruned_ci + (int64_t)b * n_prune : nullptr;
    int j0, j1;
    sels_slice(n, g, &j0, &j1);
    if (n <= n_prune) {                                     // everything survives; the last block pads
        for (int j = j0 + threadIdx.x; j < j1; j += SEL_THREADS) {
            out[j] = cb[j];
            if (out_ci) out_ci[j] = sb[j];
        }
        if (g == SELS_SPLIT - 1) {
            for (int j = n + threadIdx.x; j < n_prune; j += SEL_THREADS) {
                out[j] = -1;
                if (out_ci) out_ci[j] = INT_MIN;
            }
            if (threadIdx.x == 0) n_pruned[b] = n;
        }
        return;
    }
    const int32_t *sc = scratch + (int64_t)b * SELS_SCRATCH;
    int need_eq;
    const uint32_t thr = sels_threshold(sc, n_prune, warp_part, s_out, &need_eq);
    int run_gt = 0, run_eq = 0;
    for (int s = 0; s < g; ++s) {
        run_gt += sc[5120 + s];
        run_eq += sc[5120 + SELS_SPLIT + s];
    }
    for (int base = j0; base < j1; base += 4 * SEL_THREADS) {
        const int q0 = base + 4 * threadIdx.x;
        uint32_t u[4];
        int32_t id[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const int j = q0 + e;
            u[e] = j < j1 ? ((uint32_t)sb[j] ^ 0x80000000u) : 0u;
            id[e] = j < j1 ? cb[j] : 0;
        }
        int gt = 0, eq = 0;
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            gt += (q0 + e < j1 && u[e] > thr) ? 1 : 0;
            eq += (q0 + e < j1 && u[e] == thr) ? 1 : 0;
        }
        int total;
        const int before = sel_block_scan((gt << 16) | eq, &total, warp_part);
        int gt_before = run_gt + (before >> 16), eq_before = run_eq + (before & 0xffff);
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            if (q0 + e >= j1) break;
            const bool is_gt = u[e] > thr, is_eq = u[e] == thr;
            if (is_gt || (is_eq && eq_before < need_eq)) {
                const int pos = gt_before + (eq_before < need_eq ? eq_before : need_eq);
                out[pos] = id[e];
                if (out_ci) out_ci[pos] = (int32_t)(u[e] ^ 0x80000000u);
            }
            gt_before += is_gt ? 1 : 0;
            eq_before += is_eq ? 1 : 0;
        }
        run_gt += total >> 16;
        run_eq += total & 0xffff;
    }
    if (g == 0 && threadIdx.x == 0) n_pruned[b] = n_prune;
}

// Queries per call up to which the selection is spread over several blocks, and the scratch it needs.
bool select_split_used(const Index &ix, const Params &p) { return 4 * p.B <= ix.sm_count; }
size_t select_split_scratch_bytes(const Index &ix, const Params &p)
{
    return select_split_used(ix, p) ? sizeof(int32_t) * (size_t)p.B * SELS_SCRATCH : 0;
}

// The kernel with select_few costs where it does not come to that: its shared memory makes the SM change its split between kernels
// (140 queries of 8,184 candidates 14.3 -> 16.4 us, one short list 167.7 -> 168.9 a call), and its other path is slower (6 queries of a
// million, 9,439 wanted: 478 -> 517).  Taken where it applies to half the candidates that independent tokens would give: more than
// that are rare, and where it does apply it takes less than half the time.
bool select_few_used(const Index &ix, const Params &p)
{
    const double half = 0.5 * expected_candidates(ix, p);
    int want;
    return p.maxc >= 2 * SEL_SAMPLE && half >= SEL_SAMPLE &&
           select_few_applies(half > 2 * SEL_SAMPLE ? (int)half : 2 * SEL_SAMPLE, p.n_prune, &want);
}

// scratch: select_split_scratch_bytes() bytes, or NULL (one block per query then).  many: the lists are all the candidates, not
// a few contenders.
int launch_select(const Index &ix, const Params &p, const int32_t *cand, const int32_t *n_cand, const int32_t *ci,
                  int32_t *pruned, int32_t *n_pruned, int32_t *pruned_ci, int32_t *scratch, bool many, cudaStream_t st)
{
    // the slices must stay below 2^15 entries (two counters packed in an int) and be worth five launches
    if (scratch != nullptr && select_split_used(ix, p) && p.maxc >= 16384 && p.maxc < (int64_t)SELS_SPLIT * 32767) {
        CHIMERA_CUDA(cudaMemsetAsync(scratch, 0, select_split_scratch_bytes(ix, p), st));
        const dim3 grid(SELS_SPLIT, (unsigned)p.B);
        launch(sels_hist_kernel<0>, grid, SEL_THREADS, 0, st, n_cand, ci, p.maxc, p.n_prune, scratch);
        launch(sels_hist_kernel<1>, grid, SEL_THREADS, 0, st, n_cand, ci, p.maxc, p.n_prune, scratch);
        launch(sels_hist_kernel<2>, grid, SEL_THREADS, 0, st, n_cand, ci, p.maxc, p.n_prune, scratch);
        launch(sels_count_kernel, grid, SEL_THREADS, 0, st, n_cand, ci, p.maxc, p.n_prune, scratch);
        launch(sels_write_kernel, grid, SEL_THREADS, 0, st, cand, n_cand, ci, p.maxc, p.n_prune, scratch, pruned, n_pruned,
                                                        pruned_ci);
        CHIMERA_CUDA(cudaGetLastError());
        count_launch(SLOT_SELECT, 5);
        return CHIMERA_OK;
    }
    if (many && select_few_used(ix, p)) {
        CHIMERA_CUDA(allow_shared(select_kernel<true>, sizeof(SelFew)));
        launch(select_kernel<true>, (unsigned)p.B, SEL_THREADS, sizeof(SelFew), st, cand, n_cand, ci, p.maxc, p.n_prune, pruned,
               n_pruned, pruned_ci);
    } else {
        launch(select_kernel<false>, (unsigned)p.B, SEL_THREADS, 0, st, cand, n_cand, ci, p.maxc, p.n_prune, pruned, n_pruned, pruned_ci);
    }
    CHIMERA_CUDA(cudaGetLastError());
    count_launch(SLOT_SELECT);
    return CHIMERA_OK;
}

}  // namespace chimera
