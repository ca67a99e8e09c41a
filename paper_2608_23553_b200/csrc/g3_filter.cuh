// Shared by the two forms of the first cut's scan (g3_filter.cu: a query at a time; g3_batch_scan.cu: a batch at a time).
#pragma once
#include "g3_select.cuh"

namespace chimera {

constexpr int FILTER_BINS = 2048;         // histogram bins of sum_t e(c_t), 2^17 (one 128th) each

// e(c) in units of 2^16 from a row of the 8-bit table: S < 2^16 (u + 1), and for u = 255 S <= 2^16 * 257.  tm1[k]: the
// thresholds minus one, the even bytes of word k in tm1[k].x and the odd ones in tm1[k].y (16-bit fields), so that
// sum_i (u_i + 1 - t_i)+ = sum_i max(u_i, t_i - 1) - sum_i (t_i - 1).
template <int WORDS>
__device__ __forceinline__ int filter_row_excess(const uint4 *row, const uint2 *tm1, int sum_tm1)
{
    uint32_t acc = 0;
    int full = 0;
#pragma unroll
    for (int q = 0; q < WORDS / 4; ++q) {
        const uint4 v = __ldg(row + q);
        const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const uint2 t = tm1[4 * q + k];
            acc += __vmaxu2(w[k] & 0x00ff00ffu, t.x);
            acc += __vmaxu2((w[k] >> 8) & 0x00ff00ffu, t.y);
            full += __popc((((w[k] & 0x7f7f7f7fu) + 0x01010101u) & w[k]) & 0x80808080u);
        }
    }
    return (int)(acc & 0xffffu) + (int)(acc >> 16) - sum_tm1 + full;      // fields <= 32 * 256
}

double expected_tokens(const Index &ix, const Params &p);     // that a query's candidates hold
int launch_batch_quantum(const Index &ix, const Params &p, const Layout &L, const int32_t *table, const uint8_t *table8,
                         int us, char *ws, cudaStream_t st);
int launch_batch_scan(const Index &ix, const Params &p, const Layout &L, const int32_t *table, uint8_t *table8, int us,
                      const int32_t *n_cand, int32_t *hi0, char *ws, cudaStream_t st);

}  // namespace chimera
