// Block-wide selection helpers shared by the stage-3 kernels (blocks of SEL_THREADS threads).
#pragma once
#include "common.cuh"

namespace chimera {

constexpr int SEL_THREADS = 1024;
constexpr int CONT_BINS = 8192;         // histogram bins of coarse_key() (two keys share a bin for q_len 64)

// The histogram key of a lower bound in the contender step: floor(lo / 2^16) clamped at 0 -- a valid, slightly smaller
// lower bound (documents with an empty column fall to the bottom, which only lowers the threshold).
__device__ __forceinline__ int coarse_key(int32_t lo) { return lo < 0 ? 0 : lo >> 16; }

// Exclusive prefix sum over the block (SEL_THREADS threads); *total gets the block sum.  Two barriers.
__device__ __forceinline__ int sel_block_scan(int v, int *total, int *warp_part /* [32] */)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int incl = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        int t = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += t;
    }
    __syncthreads();                     // warp_part may still be read from a previous call
    if (lane == 31) warp_part[warp] = incl;
    __syncthreads();
    int pw = warp_part[lane];            // 32 warps
    int pincl = pw;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        int t = __shfl_up_sync(0xffffffffu, pincl, o);
        if (lane >= o) pincl += t;
    }
    *total = __shfl_sync(0xffffffffu, pincl, 31);
    int before = __shfl_sync(0xffffffffu, pincl - pw, warp);
    return before + incl - v;
}

// tau of the contender step: the smallest lower bound in the histogram bin that holds the n_prune-th largest of lb[0..n)
// (n > n_prune), so at most that one.  Whole block; hist: CONT_BINS entries, of any content.  The lower bounds are
// lo = 2^16 sum - zeros (2^24 + 2^16) with sum = the sum of nq 8-bit maxima, so coarse_key(lo) is a key of at most 14 bits and
// 2^16 key <= lo: one histogram sweep (two neighbouring keys share a bin for q_len 64) finds tau without radix passes.
__device__ __forceinline__ int contender_bin_shift(int nq) { return 255 * nq < CONT_BINS ? 0 : 1; }
__device__ __forceinline__ int32_t contender_threshold(const int32_t *__restrict__ lb, int n, int n_prune, int nq, int *hist,
                                                       int *warp_part, int *s_bin)
{
    const int bin_shift = contender_bin_shift(nq);
    for (int i = threadIdx.x; i < CONT_BINS; i += SEL_THREADS) hist[i] = 0;
    __syncthreads();
    for (int base = 0; base < n; base += 16 * SEL_THREADS) {
        int32_t v[16];
#pragma unroll
        for (int e = 0; e < 16; ++e) {
            const int j = base + e * SEL_THREADS + threadIdx.x;
            v[e] = j < n ? lb[j] : 0;
        }
#pragma unroll
        for (int e = 0; e < 16; ++e) {
            const int j = base + e * SEL_THREADS + threadIdx.x;
            if (j < n) atomicAdd(&hist[coarse_key(v[e]) >> bin_shift], 1);
        }
    }
    __syncthreads();
    // descending bins, CONT_BINS / SEL_THREADS consecutive bins per thread
    constexpr int PER = CONT_BINS / SEL_THREADS;
    const int first_bin = CONT_BINS - 1 - PER * (int)threadIdx.x;  // this thread owns first_bin, first_bin - 1, ...
    int h[PER], mine = 0;
#pragma unroll
    for (int e = 0; e < PER; ++e) { h[e] = hist[first_bin - e]; mine += h[e]; }
    int total;
    int before = sel_block_scan(mine, &total, warp_part);
    if (before < n_prune && n_prune <= before + mine) {
#pragma unroll
        for (int e = 0; e < PER; ++e) {
            if (before < n_prune && n_prune <= before + h[e]) *s_bin = first_bin - e;
            before += h[e];
        }
    }
    __syncthreads();
    return (*s_bin << bin_shift) << 16;
}

// Radix select (11 + 11 + 10 bits, most significant first) of the `want`-th largest value of sb[0..n) in the order of
// u = value ^ 0x80000000.  Needs n >= want >= 1.  Returns that value's u; *need_eq = how many entries equal to it
// belong to the top `want` (the rest of the top `want` are strictly greater).  Whole block, uniform.
template <class Load>     // load(j) = value j (int32)
__device__ __forceinline__ uint32_t radix_select(Load load, int n, int want_in, int *hist, int *warp_part,
                                                 uint32_t *s_prefix, int *s_want, int *need_eq)
{
    if (threadIdx.x == 0) { *s_prefix = 0u; *s_want = want_in; }
    const int shifts[3] = {21, 10, 0};
    const int widths[3] = {11, 11, 10};
    uint32_t known_mask = 0u;
    for (int pass = 0; pass < 3; ++pass) {
        const int shift = shifts[pass], bins = 1 << widths[pass];
        for (int i = threadIdx.x; i < 2048; i += SEL_THREADS) hist[i] = 0;
        __syncthreads();
        const uint32_t prefix = *s_prefix;
        const int want = *s_want;
        // eight independent loads per thread before their histogram updates (the loop is latency-bound otherwise)
        for (int base = 0; base < n; base += 8 * SEL_THREADS) {
            uint32_t u[8];
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                const int j = base + e * SEL_THREADS + threadIdx.x;
                u[e] = j < n ? ((uint32_t)load(j) ^ 0x80000000u) : 0u;
            }
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                const int j = base + e * SEL_THREADS + threadIdx.x;
                if (j < n && (u[e] & known_mask) == prefix) atomicAdd(&hist[(u[e] >> shift) & (bins - 1)], 1);
            }
        }
        __syncthreads();
        // descending bins: thread t owns bins (bins-1-2t) and (bins-2-2t)
        int hi_bin = bins - 1 - 2 * (int)threadIdx.x, lo_bin = hi_bin - 1;
        int h_hi = hi_bin >= 0 ? hist[hi_bin] : 0;
        int h_lo = lo_bin >= 0 ? hist[lo_bin] : 0;
        int total;
        int before = sel_block_scan(h_hi + h_lo, &total, warp_part);
        // the wanted rank falls in the first bin whose cumulative count reaches `want`
        if (before < want && want <= before + h_hi + h_lo) {
            if (want <= before + h_hi) {
                *s_prefix = prefix | ((uint32_t)hi_bin << shift);
                *s_want = want - before;
            } else {
                *s_prefix = prefix | ((uint32_t)lo_bin << shift);
                *s_want = want - before - h_hi;
            }
        }
        known_mask |= (uint32_t)(bins - 1) << shift;
        __syncthreads();
    }
    *need_eq = *s_want;
    return *s_prefix;
}

}  // namespace chimera
