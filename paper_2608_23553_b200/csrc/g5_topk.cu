// Stage 5: batched top-k (Definition 2, Eq. 1): per query the k survivors with the largest stage-4 score, best
// first, ties towards the smaller document id; missing entries are (-1, -inf).
//
// One block per query.  Each (score, id) becomes a 64-bit key whose unsigned order is (score desc, id asc); the keys
// are sorted descending with a bitonic network in shared memory (n_prune <= 16384 keys = 128 KB) and the first k are
// decoded back -- only those that reach the k-th score, found by a radix select, when k is at most a quarter of them.
// For k <= 16 the keys stay in registers instead: each warp extracts its own k largest, one after the other with hardware maxima
// over the warp, and one warp merges those lists, so there is one barrier in all (the block extracting its maximum k times took
// two per result: one query of 256 entries and k = 10 6.7 us, 3.2 so; 256 queries of 1,024 10.3, 5.8).
#include <math.h>

#include "g3_select.cuh"

namespace chimera {

constexpr int TOPK_THREADS = 1024;

__device__ __forceinline__ uint32_t float_order(float f)
{
    uint32_t u = __float_as_uint(f);
    if (u == 0x80000000u) u = 0u;        // -0 and +0 are the same score (the tie goes to the smaller id)
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
__device__ __forceinline__ float float_unorder(uint32_t o)
{
    uint32_t u = (o & 0x80000000u) ? (o & 0x7fffffffu) : ~o;
    return __uint_as_float(u);
}

// Entry j of query b.  A query's entries are one run of n_prune (seg_len = n_prune) or, for the merge of several
// shards' lists laid out [shard][query][seg_len], one run of seg_len per shard, seg_stride apart.
__device__ __forceinline__ int64_t entry_index(int j, int b, int seg_len, long long seg_stride)
{
    return (int64_t)(j / seg_len) * seg_stride + (int64_t)b * seg_len + j % seg_len;
}

// Descending bitonic sort of n_pow2 keys in shared memory; whole block.
__device__ __forceinline__ void bitonic_sort(unsigned long long *keys, int n_pow2)
{
    for (int size = 2; size <= n_pow2; size <<= 1) {
        for (int stride = size >> 1; stride > 0; stride >>= 1) {
            for (int t = threadIdx.x; t < (n_pow2 >> 1); t += TOPK_THREADS) {
                int lo = 2 * t - (t & (stride - 1));      // index with the stride bit clear
                int hi = lo + stride;
                bool descending = (lo & size) == 0;
                unsigned long long a = keys[lo], c = keys[hi];
                if ((a < c) == descending) { keys[lo] = c; keys[hi] = a; }
            }
            __syncthreads();
        }
    }
}

// SELECT (at least four times as many entries as wanted): the k-th largest score by radix select, then only the entries
// that reach it are sorted (16,384 entries, k = 1,000: 185 us for sorting all, 41 with the selection; 1,024 and k = 20:
// 16.4 us for sorting runs in registers and merging them, 12.4 so).  More ties at that
// score than the second array holds: everything is sorted after all.
template <bool SELECT>
__global__ void __launch_bounds__(TOPK_THREADS)
topk_kernel(const int32_t *__restrict__ pruned, const float *__restrict__ score4, int n_prune, int n_pow2, int cap, int k,
            int seg_len, long long seg_stride, int32_t *__restrict__ out_ids, float *__restrict__ out_scores)
{
    pdl_entry();
    extern __shared__ unsigned long long topk_keys[];
    unsigned long long *keys = topk_keys;
    const int b = blockIdx.x;
    for (int j = threadIdx.x; j < n_pow2; j += TOPK_THREADS) {
        unsigned long long key = 0ull;
        if (j < n_prune) {
            const int64_t at = entry_index(j, b, seg_len, seg_stride);
            int32_t id = pruned[at];
            if (id >= 0)
                key = ((unsigned long long)float_order(score4[at]) << 32) | (uint32_t)(0xFFFFFFFFu - (uint32_t)id);
        }
        keys[j] = key;
    }
    __syncthreads();
    if (SELECT) {
        __shared__ int hist[2048];
        __shared__ int warp_part[32];
        __shared__ uint32_t s_prefix;
        __shared__ int s_want, s_count;
        if (threadIdx.x == 0) s_count = 0;
        int need_eq;
        const uint32_t thr = radix_select([&](int j) { return (int)((uint32_t)(keys[j] >> 32) ^ 0x80000000u); }, n_prune, k, hist,
                                          warp_part, &s_prefix, &s_want, &need_eq);
        unsigned long long *best = keys + n_pow2;         // room for 2 * pow2(k)
        for (int j = threadIdx.x; j < n_prune; j += TOPK_THREADS)
            if ((uint32_t)(keys[j] >> 32) >= thr) {
                const int at = atomicAdd(&s_count, 1);
                if (at < cap) best[at] = keys[j];
            }
        __syncthreads();
        const int cnt = s_count;
        if (cnt <= cap) {
            int m = 2;
            while (m < cnt) m <<= 1;
            for (int j = cnt + threadIdx.x; j < m; j += TOPK_THREADS) best[j] = 0ull;
            __syncthreads();
            bitonic_sort(best, m);
            keys = best;
            n_pow2 = m;
        } else {
            bitonic_sort(keys, n_pow2);
        }
    } else {
        bitonic_sort(keys, n_pow2);
    }
    for (int r = threadIdx.x; r < k; r += TOPK_THREADS) {
        unsigned long long key = r < n_pow2 ? keys[r] : 0ull;
        if (key == 0ull) {
            out_ids[(int64_t)b * k + r] = -1;
            out_scores[(int64_t)b * k + r] = -INFINITY;
        } else {
            out_ids[(int64_t)b * k + r] = (int32_t)(0xFFFFFFFFu - (uint32_t)key);
            out_scores[(int64_t)b * k + r] = float_unorder((uint32_t)(key >> 32));
        }
    }
}

// Largest key of the warp.
__device__ __forceinline__ unsigned long long warp_max_key(unsigned long long key)
{
    const uint32_t hi = (uint32_t)(key >> 32), most = __reduce_max_sync(0xffffffffu, hi);
    const uint32_t low = __reduce_max_sync(0xffffffffu, hi == most ? (uint32_t)key : 0u);
    return (unsigned long long)most << 32 | low;
}

constexpr int TOPK_FEW = 16;      // largest k of this kernel
template <int KPT>                // keys per thread: n_prune <= KPT * blockDim.x
__global__ void __launch_bounds__(TOPK_THREADS)
topk_small_kernel(const int32_t *__restrict__ pruned, const float *__restrict__ score4, int n_prune, int k,
                  int seg_len, long long seg_stride, int32_t *__restrict__ out_ids, float *__restrict__ out_scores)
{
    pdl_entry();
    __shared__ unsigned long long s_best[32][TOPK_FEW];      // of each warp, descending
    const int b = blockIdx.x, lane = threadIdx.x & 31, warp = threadIdx.x >> 5, warps = blockDim.x >> 5;
    unsigned long long keys[KPT];
#pragma unroll
    for (int e = 0; e < KPT; ++e) {
        const int j = e * blockDim.x + threadIdx.x;
        keys[e] = 0ull;
        if (j < n_prune) {
            const int64_t at = entry_index(j, b, seg_len, seg_stride);
            const int32_t id = pruned[at];
            const float score = score4[at];
            if (id >= 0) keys[e] = ((unsigned long long)float_order(score) << 32) | (uint32_t)(0xFFFFFFFFu - (uint32_t)id);
        }
    }
    for (int r = 0; r < k; ++r) {
        unsigned long long m = keys[0];
#pragma unroll
        for (int e = 1; e < KPT; ++e) m = keys[e] > m ? keys[e] : m;
        m = warp_max_key(m);                                 // (keys are distinct, the id is part of them: one owner)
#pragma unroll
        for (int e = 0; e < KPT; ++e)
            if (keys[e] == m) keys[e] = 0ull;
        if (lane == 0) s_best[warp][r] = m;
    }
    __syncthreads();
    if (warp > 0) return;
    int next = 0;                                            // lane = list: the first of its entries that is still there
    unsigned long long mine = lane < warps ? s_best[lane][0] : 0ull, result = 0ull;
    for (int r = 0; r < k; ++r) {
        const unsigned long long m = warp_max_key(mine);
        if (lane == r) result = m;
        if (m != 0ull && mine == m) mine = ++next < k ? s_best[lane][next] : 0ull;
    }
    if (lane < k) {
        out_ids[(int64_t)b * k + lane] = result ? (int32_t)(0xFFFFFFFFu - (uint32_t)result) : -1;
        out_scores[(int64_t)b * k + lane] = result ? float_unorder((uint32_t)(result >> 32)) : -INFINITY;
    }
}

// n entries per query (laid out by entry_index) -> the best k.
static int launch_topk_entries(const int32_t *ids, const float *scores, int B, int n, int k, int seg_len,
                               long long seg_stride, int32_t *out_ids, float *out_scores, cudaStream_t st)
{
    if (k <= TOPK_FEW && n <= 16 * TOPK_THREADS) {
        const int threads = n >= TOPK_THREADS ? TOPK_THREADS : (n + 31) / 32 * 32;
        launch(n <= TOPK_THREADS       ? topk_small_kernel<1>
               : n <= 4 * TOPK_THREADS ? topk_small_kernel<4>
                                       : topk_small_kernel<16>,
               (unsigned)B, threads, 0, st, ids, scores, n, k, seg_len, seg_stride, out_ids, out_scores);
        CHIMERA_CUDA(cudaGetLastError());
        return CHIMERA_OK;
    }
    int n_pow2 = 2;
    while (n_pow2 < n) n_pow2 <<= 1;
    const size_t smem = sizeof(unsigned long long) * (size_t)n_pow2;
    constexpr size_t TOPK_SMEM = 128 * 1024;
    if (smem > TOPK_SMEM) return fail(CHIMERA_UNSUPPORTED, "top-k over %d entries per query does not fit shared memory", n);
    int cap = 4;
    while (cap < 2 * k) cap <<= 1;
    const bool select = n >= 4 * k && n >= 256;
    const size_t bytes = smem + (select ? sizeof(unsigned long long) * (size_t)cap : 0);
    auto kern = select ? topk_kernel<true> : topk_kernel<false>;
    if (bytes > 48 * 1024 - 16 * 1024)                    // (the selection has 8 KB of its own)
        CHIMERA_CUDA(allow_shared(kern, TOPK_SMEM + (select ? TOPK_SMEM / 2 : 0)));     // (k <= n / 4, so cap <= n_pow2 / 2)
    launch(kern, (unsigned)B, TOPK_THREADS, bytes, st, ids, scores, n, n_pow2, cap, k, seg_len, seg_stride, out_ids, out_scores);
    CHIMERA_CUDA(cudaGetLastError());
    return CHIMERA_OK;
}

int launch_topk(const Index &ix, const Params &p, const int32_t *pruned, const float *score4, int32_t *out_ids,
                float *out_scores, cudaStream_t st)
{
    (void)ix;
    const int rc = launch_topk_entries(pruned, score4, p.B, p.n_prune, p.k, p.n_prune, 0, out_ids, out_scores, st);
    if (rc) return rc;
    count_launch(SLOT_TOPK);
    return CHIMERA_OK;
}

// Final merge of a document-sharded search: all_ids / all_scores are the shards' top-k lists, [world][B][k] (global
// ids, -1 / -inf padded); out = the best k of their union per query, (score desc, id asc).
int launch_shard_merge_topk(const int32_t *all_ids, const float *all_scores, int world, int B, int k, int32_t *out_ids,
                            float *out_scores, cudaStream_t st)
{
    const int rc = launch_topk_entries(all_ids, all_scores, B, world * k, k, k, (long long)B * k, out_ids, out_scores, st);
    if (rc) return rc;
    count_launch(SLOT_TOPK);
    return CHIMERA_OK;
}

}  // namespace chimera
