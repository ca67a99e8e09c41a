// Stage 1: score table S[c, i] = <q_i, centroid_c> for every query token and every centroid (Definition 1's inner
// product), evaluated exactly in integers:
//     Xq = rint(q * 2^22), Xc = rint(c * 2^22),  T = sum_d Xq[d] * Xc[d],  S = floor((T + 2^19) / 2^20)   (Q.24).
// Each 23-bit integer is split into three balanced base-256 digits, so T = sum_{a,b} 256^(a+b) P_ab with the nine
// digit-plane products P_ab = sum_d qa[d] * cb[d] being int8 x int8 -> int32 contractions (exact in any order).
// Products of equal weight a+b share an accumulator (five accumulators, each |.| < 2^23); the epilogue recombines
// them with shifts (in 32-bit arithmetic, see combine_digits) and rounds.
//
// The contraction runs on the 5th-generation tensor cores: tcgen05.mma kind::i8 (int8 operands, int32 accumulators in
// tensor memory), M = 128 centroids, K = 32 dimensions per instruction.  One CTA owns a tile of 128 centroids for its
// whole life and keeps their three digit planes IN TENSOR MEMORY (the A operand of the instruction is read from there:
// lane = centroid, 32 bytes per K step), so only the query digits come from shared memory and the 48 KB that the tile
// would take there go to a deeper pipeline of query tiles.  A query tile is 32 query-token rows; its three digit planes
// are K-major rows with a 128-byte pitch (dimensions beyond D are zero), brought into 128-byte-swizzled shared memory
// one after the other by TMA (one plain per-CTA cp.async.bulk.tensor load per tile, no multicast), four tiles deep, so
// that one instruction with N = 96 multiplies a centroid digit plane with all three query planes (see the schedule at
// the MMA loop).  Tensor memory per CTA: 5 accumulators x 32 columns + 96 columns of centroid digits = 256 columns, so
// two CTAs share an SM.  A producer warp issues the loads and the MMAs; eight warps drain the accumulators (two per
// tensor-memory lane quarter; how they share it depends on whether the scores are stored).  A draining warp hands the accumulators
// back as soon as its tcgen05.ld's have landed in registers, so the next tile's MMAs run while it recombines and stores.  An
// isolated loop of these instructions runs at half a cycle per column of N (8,192 multiply-adds per SM cycle) but
// never faster than ~45 cycles per instruction, which is why the instructions here are N = 96 wide (48 cycles).
// Every wait on an mbarrier is bounded; a wait that gives up sets the workspace's TIMEOUT status bit, and the CTA
// waits (bounded) for its loads in flight, frees its tensor memory and returns.
#include <cuda.h>

#include "common.cuh"
#include "umma.cuh"

namespace chimera {

constexpr int G1_M = 128;            // centroids per tile (MMA M)
constexpr int G1_N = 32;             // query-token rows per tile (MMA N)
constexpr int G1_ROW_BYTES = 128;    // digit-plane row pitch = padded dimension count
constexpr int G1_WPQ = 2;            // draining warps per tensor-memory lane quarter
constexpr int G1_DRAIN_WARPS = 4 * G1_WPQ;
constexpr int G1_THREADS = 32 * (G1_DRAIN_WARPS + 1);      // + the producer warp
constexpr int G1_STAGES = 4;         // query tiles in flight
constexpr int G1_TMEM_COLS = 256;
constexpr int G1_ACC_COLS = 5 * G1_N;                      // accumulators in columns [0, 160)
constexpr int G1_A_COL = G1_ACC_COLS;                      // centroid digits in columns [160, 256): 32 per plane
constexpr uint32_t G1_B_PLANE = G1_N * G1_ROW_BYTES;       // 4 KB
constexpr uint32_t G1_B_LOAD = 3 * G1_B_PLANE;             // 12 KB: the three digit planes of a tile, one after the other
constexpr uint32_t G1_B_STAGE = 5 * G1_B_PLANE;            // 20 KB: + 64 rows of zeros (see the MMA schedule)
constexpr uint32_t G1_SMEM = G1_STAGES * G1_B_STAGE + 1024 /* alignment slack */ + 64 /* barriers */;
static_assert(G1_ACC_COLS + 96 <= G1_TMEM_COLS, "accumulators and centroid digits share the allocation");

// floor((T + 2^19) / 2^20) with T = a0 + 2^8 a1 + 2^16 a2 + 2^24 a3 + 2^32 a4, in 32-bit arithmetic.  Split T as
// u + 2^16 v with u = a0 + 2^8 a1 (|a0| < 2^23, |a1| < 2^23: no overflow) and
// v = a2 + 2^8 a3 + 2^16 a4.  v is about T / 2^16, which fits 32 bits whenever the result does (|S| < 2^31 means
// |T| < 2^51; here |T| < 2^45), so computing it modulo 2^32 loses nothing.  Nested floor divisions compose:
// floor((x + 2^16 v) / 2^20) = floor((floor(x / 2^16) + v) / 2^4) for any integers x, v; arithmetic right shifts are
// floor divisions.
__device__ __forceinline__ int32_t combine_digits(int32_t a0, int32_t a1, int32_t a2, int32_t a3, int32_t a4)
{
    const int32_t u = a0 + (a1 << 8);
    const int32_t v = a2 + (int32_t)((uint32_t)a3 << 8) + (int32_t)((uint32_t)a4 << 16);
    return ((u >> 16) + v + 8) >> 4;                    // the rounding constant is a multiple of 2^16
}

__device__ __forceinline__ void mbar_arrive(uint32_t bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}

// Which centroid tiles a launch covers, and whether it feeds the probe stage (FILTER).
//   tile_stride == 0: every tile (tile = blockIdx.x).
//   tile_stride  > 1, sample != 0: the sample tiles 0, s, 2s, ... (tile = blockIdx.x * s).
//   tile_stride  > 1, sample == 0: all the others (the j-th tile that is not a multiple of s).
// FILTER (only with the "others"): thr[row] holds, for every query-token row, a lower bound on the score of the row's
// nprobe-th best centroid (found on the sample; padded to whole tiles of rows); every score >= thr[row] goes, as a (score,
// centroid) key, into that row's queue (keys[row][cap], counted in cnt[row]; entries past cap are dropped and the count tells).  The top nprobe
// of a row are then in its queue, so the probe stage never reads the table again, and a search that needs only the
// probes passes no table (the RaBitQ pipeline: 2.1 GB less to write at Mid, batch 256).
// redo: a flag per query (nonzero: its rows of these tiles are wanted after all); a CTA without such a query returns.
struct G1Tiles {
    int tile_stride, sample;
    const int32_t *thr;
    int32_t *cnt;
    unsigned long long *keys;
    int cap;
    const int32_t *redo;
};

// grid (centroid tiles of the launch, n_splits).  Each CTA: one centroid tile, query-row tiles
// [blockIdx.y * tiles_per_split, ...).  KS = D / 32 MMA steps per digit-plane product.
template <int KS, bool FILTER, bool TABLE>
__global__ void __launch_bounds__(G1_THREADS, 2)
score_table_umma(const int8_t *__restrict__ cdig, const __grid_constant__ CUtensorMap map_q, int64_t K, int nq,
                 int64_t q_rows, int n_tiles, int tiles_per_split, int32_t *__restrict__ table,
                 uint8_t *__restrict__ table8, uint32_t *status, long long wait_limit, int skip_loads, G1Tiles tiles)
{
    extern __shared__ uint8_t smem_raw[];
    __shared__ uint32_t s_tmem_base;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    int c_tile = (int)blockIdx.x;
    if (tiles.tile_stride > 1)
        c_tile = tiles.sample ? c_tile * tiles.tile_stride : c_tile + c_tile / (tiles.tile_stride - 1) + 1;
    const int64_t c0 = (int64_t)c_tile * G1_M;
    // The centroid tile's digit planes, lane = centroid: plane h = warp / 4 of 0, 1 and half h of plane 2 for each of the eight
    // draining warps.  All twelve loads are on their way before anything else, the wait for the kernel before included (the
    // index does not come from it): one query leaves a CTA a single tile, whose time is mostly
    // this latency (plane after plane by four warps, behind the set-up: Large 48.8 us, now 47.0; 256 queries 3.19, now 3.07 ms).
    uint4 a[12];
    auto load_centroids = [&]() {
        const int64_t c = c0 + (warp & 3) * 32 + lane;
        const int h = warp >> 2;
        const uint4 *full = reinterpret_cast<const uint4 *>(cdig + ((int64_t)h * K + c) * G1_ROW_BYTES);
        const uint4 *part = reinterpret_cast<const uint4 *>(cdig + (2 * K + c) * G1_ROW_BYTES) + 4 * h;
#pragma unroll
        for (int x = 0; x < 12; ++x) {
            a[x] = make_uint4(0u, 0u, 0u, 0u);
            if (warp < G1_DRAIN_WARPS && c < K) a[x] = __ldg(x < 8 ? full + x : part + x - 8);
        }
    };
    if (FILTER || tiles.redo == nullptr) load_centroids();
    pdl_entry();
    const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    const uint32_t sB = base;                                  // G1_STAGES x (3 planes x 4 KB + 8 KB of zeros)
    const uint32_t bars = sB + G1_STAGES * G1_B_STAGE;
    const uint32_t bar_full = bars;                            // [G1_STAGES]: a query tile has landed
    const uint32_t bar_mma = bars + 8 * G1_STAGES;             // a tile's accumulators are complete
    const uint32_t bar_empty = bar_mma + 8;                    // every draining warp has the accumulators in registers
    const int t_begin = blockIdx.y * tiles_per_split;
    int t_end = t_begin + tiles_per_split;
    if (t_end > n_tiles) t_end = n_tiles;
    const int my_tiles = t_end > t_begin ? t_end - t_begin : 0;
    if (!FILTER && tiles.redo != nullptr) {
        const int64_t r_end = (int64_t)t_end * G1_N < q_rows ? (int64_t)t_end * G1_N : q_rows;
        int wanted = 0;
        if (my_tiles > 0)
            for (int64_t b = (int64_t)t_begin * G1_N / nq + tid; b <= (r_end - 1) / nq; b += G1_THREADS) wanted |= tiles.redo[b];
        if (!__syncthreads_or(wanted)) return;
        load_centroids();
    }

    if (tid == 0) {
        for (int s = 0; s < G1_STAGES; ++s) mbar_init(bar_full + 8 * s, 1);
        mbar_init(bar_mma, 1);
        mbar_init(bar_empty, G1_DRAIN_WARPS);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        __syncwarp();
        tmem_alloc(&s_tmem_base, G1_TMEM_COLS);
    }
    // the 64 zero rows behind each stage's planes (the loads never touch them); only the stages this CTA will use
    const uint32_t used_stages = my_tiles < G1_STAGES ? (uint32_t)my_tiles : (uint32_t)G1_STAGES;
    for (uint32_t e = tid; e < used_stages * (G1_B_STAGE - G1_B_LOAD) / 16; e += G1_THREADS) {
        const uint32_t per = (G1_B_STAGE - G1_B_LOAD) / 16;
        const uint32_t addr = sB + (e / per) * G1_B_STAGE + G1_B_LOAD + (e % per) * 16;
        asm volatile("st.shared.v4.b32 [%0], {%1, %1, %1, %1};" ::"r"(addr), "r"(0u) : "memory");
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");     // visible to the tensor core's reads
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = s_tmem_base;

    // the first query tiles are requested before the centroid tile is fetched, so the two latencies overlap.
    // skip_loads (test hook): no load is issued and no bytes are expected, so the producer's first wait runs into its
    // limit with nothing in flight
    int issued = 0;                                            // producer thread: tiles whose load has been issued
    auto load_tile = [&](int it) {
        const uint32_t bar = bar_full + 8 * (it % G1_STAGES);
        mbar_expect_tx(bar, G1_B_LOAD);
        tma_load_3d(sB + (it % G1_STAGES) * G1_B_STAGE, &map_q, 0, (t_begin + it) * G1_N, 0, bar);
    };
    if (warp == G1_DRAIN_WARPS && lane == 0 && !skip_loads)
        for (; issued < my_tiles && issued < G1_STAGES; ++issued) load_tile(issued);

    // ---- the centroid tile's digit planes into tensor memory (a warp reaches its own lane quarter, warp % 4) ----------
    if (warp < G1_DRAIN_WARPS) {
        const uint32_t lane_addr = tmem + ((uint32_t)((warp & 3) * 32) << 16) + G1_A_COL;
        const int h = warp >> 2;
        uint32_t full[32], part[16];
#pragma unroll
        for (int x = 0; x < 8; ++x) {
            full[4 * x] = a[x].x; full[4 * x + 1] = a[x].y; full[4 * x + 2] = a[x].z; full[4 * x + 3] = a[x].w;
        }
#pragma unroll
        for (int x = 0; x < 4; ++x) {
            part[4 * x] = a[8 + x].x; part[4 * x + 1] = a[8 + x].y; part[4 * x + 2] = a[8 + x].z; part[4 * x + 3] = a[8 + x].w;
        }
        tmem_st(lane_addr + h * 32, full);
        tmem_st(lane_addr + 64 + h * 16, part);
        asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();

    // instruction descriptors: D = S32, A and B signed 8-bit, both K-major, M = 128, N = 96 or 160
    constexpr uint32_t IDESC_BASE = (2u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(G1_M >> 4) << 24);
    constexpr uint32_t IDESC_3 = IDESC_BASE | ((uint32_t)((3 * G1_N) >> 3) << 17);
    constexpr uint32_t IDESC_5 = IDESC_BASE | ((uint32_t)((5 * G1_N) >> 3) << 17);

    if (warp == G1_DRAIN_WARPS) {
        // ================================================================================= producer (one thread) ===
        if (lane == 0) {
            bool ok = true;
            int it = 0;
            for (; it < my_tiles; ++it) {
                const int stage = it % G1_STAGES;
                ok = mbar_wait(bar_full + 8 * stage, (it / G1_STAGES) & 1, wait_limit);
                // the previous tile's accumulators are in the draining warps' registers: its MMAs are complete (so
                // its stage of query digits is free) and tensor memory may be overwritten
                if (ok && it > 0) ok = mbar_wait(bar_empty, (it - 1) & 1, wait_limit);
                if (!ok) break;
                tc_fence_after();
                // The stage holds the query's digit planes a = 0, 1, 2 as 96 consecutive B rows, and the accumulators
                // of weight w = 0..4 are consecutive groups of 32 columns.  One instruction with the centroids' digit
                // plane b as A and all 96 rows as B therefore adds the products of weight b, b + 1, b + 2 to the
                // accumulators starting at column 32 b: three instructions of N = 96 per K step instead of nine of
                // N = 32 (an instruction takes N / 2 cycles but at least ~45: -8 % on the whole kernel).  The very
                // first instruction runs over 160 rows (the last 64 are zeros) without accumulating, which clears
                // weights 3 and 4.
                const uint64_t db0 = umma_desc(sB + stage * G1_B_STAGE);
#pragma unroll
                for (int k = 0; k < KS; ++k) {
#pragma unroll
                    for (int bdig = 0; bdig < 3; ++bdig) {     // centroid digit
                        if (k == 0 && bdig == 0)
                            umma_i8_ts(tmem, tmem + G1_A_COL, db0, IDESC_5, 0u);
                        else
                            umma_i8_ts(tmem + bdig * G1_N, tmem + G1_A_COL + bdig * 32 + 8 * k, db0 + (uint64_t)(2 * k),
                                       IDESC_3, 1u);
                    }
                }
                umma_commit(bar_mma);
                // refill the stage that the previous tile used
                if (it > 0 && issued < my_tiles && !skip_loads) {
                    load_tile(issued);                         // issued == it - 1 + G1_STAGES: the same stage
                    ++issued;
                }
            }
            if (!ok) {
                atomicOr(status, ST_TIMEOUT);
                // loads in flight write this CTA's shared memory: wait for them (bounded) before leaving
                if (!skip_loads)
                    for (int j = it; j < issued; ++j)
                        mbar_wait(bar_full + 8 * (j % G1_STAGES), (j / G1_STAGES) & 1, wait_limit);
            } else if (my_tiles > 0) {
                // the last tile's MMAs read shared memory and tensor memory: complete before the CTA leaves
                if (!mbar_wait(bar_mma, (my_tiles - 1) & 1, wait_limit)) atomicOr(status, ST_TIMEOUT);
            }
        }
    } else {
        // ============================================================================================ draining warps ===
        const uint32_t unq = (uint32_t)nq, n_rows = (uint32_t)q_rows, n_cent = (uint32_t)K;
        unsigned long long pend_key = 0ull, *pend_dst = nullptr;   // FILTER: this thread's last key, not stored yet
        int pend_slot = 0;
        // The slot comes back from the atomic hundreds of cycles later; the key is stored only when this thread's next key
        // turns up (or at the end), so nobody waits for it.
        auto push = [&](uint32_t row, uint32_t c, int32_t v) {
            if (pend_key && pend_slot < tiles.cap) pend_dst[pend_slot] = pend_key;
            pend_key = key_int(v, (int32_t)c);
            pend_dst = tiles.keys + (int64_t)row * tiles.cap;
            pend_slot = atomicAdd(tiles.cnt + row, 1);
        };
        // (the vote makes the decision uniform: the tensor-memory loads below need the whole warp)
        auto wait_tile = [&](int it) {
            const bool ok = __all_sync(0xffffffffu, mbar_wait(bar_mma, it & 1, wait_limit));
            if (ok) tc_fence_after();
            else if (lane == 0) atomicOr(status, ST_TIMEOUT);
            return ok;
        };
        auto hand_back = [&]() {                               // the accumulators may be overwritten from here on
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(bar_empty);
        };
        if (!TABLE) {
            // Only the keys are wanted, and issue binds.  Warp w reads tensor-memory lanes 32 (w % 4) ... + 31 (a centroid a
            // thread) and the 16 columns from 16 (w / 4) on: column 8 o + 2 g + b is row 8 g + 2 o + b of the tile (table_row()).
            // Passing rows as a mask and one push in a loop: copies of the push cost the warp whenever a single lane takes one (stage 1 of
            // 256 queries, 8,300 centroids 226 us so and 302 with copies, 17,000 307 and 370, 65,536 677 and 679 to 696).  Both halves are
            // combined before either is looked at (one after the other 96 registers and spills: 685).  Rows past the end have the
            // largest threshold.
            const uint32_t c = (uint32_t)c0 + (warp & 3) * 32 + lane;
            const int group = warp >> 2;
            const uint32_t lane_addr = tmem + ((uint32_t)((warp & 3) * 32) << 16) + 16 * group;
            for (int it = 0; it < my_tiles; ++it) {
                const uint32_t r0 = (uint32_t)(t_begin + it) * G1_N + 4 * group;
                int32_t thr_v[16];                             // by column; the same for every lane, asked for before the wait
#pragma unroll
                for (int g = 0; g < 4; ++g) {
                    const int4 v = __ldg(reinterpret_cast<const int4 *>(tiles.thr + r0 + 8 * g));
                    thr_v[2 * g] = v.x; thr_v[2 * g + 1] = v.y; thr_v[8 + 2 * g] = v.z; thr_v[8 + 2 * g + 1] = v.w;
                }
                if (!wait_tile(it)) break;
                int32_t accs[2][5][8];
#pragma unroll
                for (int w = 0; w < 5; ++w) {
                    tmem_ld8(lane_addr + w * G1_N, accs[0][w]);
                    tmem_ld8(lane_addr + w * G1_N + 8, accs[1][w]);
                }
                tmem_ld_wait();
                hand_back();
                int32_t out[2][8];
#pragma unroll
                for (int o = 0; o < 2; ++o)
#pragma unroll
                    for (int x = 0; x < 8; ++x)
                        out[o][x] = combine_digits(accs[o][0][x], accs[o][1][x], accs[o][2][x], accs[o][3][x], accs[o][4][x]);
#pragma unroll
                for (int o = 0; o < 2; ++o) {
                    bool any = false;
#pragma unroll
                    for (int x = 0; x < 8; ++x) any |= out[o][x] >= thr_v[8 * o + x];
                    if (any && c < n_cent) {
                        uint32_t pass = 0u;
#pragma unroll
                        for (int x = 0; x < 8; ++x) pass |= out[o][x] >= thr_v[8 * o + x] ? 1u << x : 0u;
                        while (pass) {
                            const int x = __ffs(pass) - 1;
                            pass &= pass - 1;
                            int32_t v = out[o][0];
#pragma unroll
                            for (int y = 1; y < 8; ++y) v = x == y ? out[o][y] : v;
                            push(r0 + 8 * (x >> 1) + 2 * o + (x & 1), c, v);
                        }
                    }
                }
            }
        } else {
            // Warp w reads tensor-memory lanes 32 (w % 4) + 16 (w / 4) ... + 15 and all 32 columns: a thread gets eight
            // neighbouring query-token rows (table_row()) of two centroids, and a warp's store is a kilobyte in a row at 32 tokens.
            // With a thread per centroid and 16 rows a store was 32 pieces of 32 lines, and the stores' wavefronts (65 % of the
            // unit's) were what bound the kernel.  Mid, batch 256: 772 -> 685 us; 262,144 centroids 2,857 -> 2,533.
            // 16 columns at a time: all 32 at once need the thresholds loaded late for want of registers (702 us).
            const uint32_t c_first = (uint32_t)c0 + (warp & 3) * 32 + (warp >> 2) * 16 + (lane >> 2);      // and c_first + 8
            const uint32_t lane_addr = tmem + ((uint32_t)((warp & 3) * 32 + (warp >> 2) * 16) << 16);
            for (int it = 0; it < my_tiles; ++it) {
                const uint32_t rc = (uint32_t)(t_begin + it) * G1_N + 8 * (lane & 3);          // this thread's first query-token row
                // FILTER: the thresholds of its eight rows, asked for before the wait
                int32_t thr_v[8];
                if (FILTER) {
#pragma unroll
                    for (int g = 0; g < 2; ++g) {
                        // (rows past the end: 0x7fffffff, in the padding behind the bounds)
                        const int4 v = __ldg(reinterpret_cast<const int4 *>(tiles.thr + rc) + g);
                        thr_v[4 * g] = v.x; thr_v[4 * g + 1] = v.y; thr_v[4 * g + 2] = v.z; thr_v[4 * g + 3] = v.w;
                    }
                }
                if (!wait_tile(it)) break;
                int32_t scores[2][8];                              // of the two centroids
#pragma unroll
                for (int o = 0; o < 2; ++o) {
                    int32_t accs[5][8];
#pragma unroll
                    for (int w = 0; w < 5; ++w) tmem_ld_16x16(lane_addr + w * G1_N + 16 * o, accs[w]);
                    tmem_ld_wait();
                    if (o == 1) hand_back();
#pragma unroll
                    for (int x = 0; x < 8; ++x)
                        scores[x >> 1 & 1][4 * o + (x >> 2) * 2 + (x & 1)] =
                            combine_digits(accs[0][x], accs[1][x], accs[2][x], accs[3][x], accs[4][x]);
                }

                // (query, token) coordinates of the first row (rows fit 32 bits: n_queries * q_len < 2^23)
                const uint32_t qb0 = rc / unq, qi0 = rc - qb0 * unq;
#pragma unroll
                for (int half = 0; half < 2; ++half) {
                    const uint32_t c = c_first + 8 * half;
                    const int32_t (&out)[8] = scores[half];
                    if (FILTER && c < n_cent) {
                        bool any = false;
#pragma unroll
                        for (int e = 0; e < 8; ++e) any |= out[e] >= thr_v[e];
                        if (any) {                  // about nprobe x tile_stride keys per row in all: one lane of a warp every
                                                    // few chunks, and then hardly ever two values of the lane
                            uint32_t pass = 0u;
#pragma unroll
                            for (int e = 0; e < 8; ++e) pass |= out[e] >= thr_v[e] ? 1u << e : 0u;
                            while (pass) {
                                const int e = __ffs(pass) - 1;
                                pass &= pass - 1;
                                int32_t v = out[0];
#pragma unroll
                                for (int x = 1; x < 8; ++x) v = e == x ? out[x] : v;
                                push(rc + e, c, v);
                            }
                        }
                    }
                    if (c < n_cent && rc < n_rows) {
                        uint32_t qb = qb0, qi = qi0;
                        const int64_t at = ((int64_t)qb * K + c) * nq + qi;
                        if (table8 != nullptr) {
                            // coarse copy for the bound phase of stage 3: clamp(S >> 16, 0, 255); q_len is a multiple of 16 here,
                            // so the eight rows belong to one query
                            uint32_t w8[2];
#pragma unroll
                            for (int g = 0; g < 2; ++g) {
                                uint32_t v[4];
#pragma unroll
                                for (int e = 0; e < 4; ++e) v[e] = (uint32_t)__vimin_s32_relu(out[4 * g + e] >> 16, 255);
                                w8[g] = __byte_perm(__byte_perm(v[0], v[1], 0x0040), __byte_perm(v[2], v[3], 0x0040), 0x5410);
                            }
                            *reinterpret_cast<uint2 *>(table8 + at) = make_uint2(w8[0], w8[1]);
                        }
                        if ((nq & 7) == 0) {
                            // eight consecutive tokens of one query, 32-byte aligned: one store
                            asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(table + at),
                                         "r"(out[0]), "r"(out[1]), "r"(out[2]), "r"(out[3]), "r"(out[4]), "r"(out[5]),
                                         "r"(out[6]), "r"(out[7])
                                         : "memory");
                        } else if ((nq & 3) == 0) {
#pragma unroll
                            for (int e = 0; e < 8; e += 4) {
                                if (rc + e < n_rows)                          // q_rows is a multiple of 4 here
                                    *reinterpret_cast<int4 *>(table + ((int64_t)qb * K + c) * nq + qi) =
                                        make_int4(out[e], out[e + 1], out[e + 2], out[e + 3]);
                                qi += 4;
                                if (qi >= unq) { qi -= unq; ++qb; }           // groups of four never straddle two queries
                            }
                        } else {
#pragma unroll
                            for (int e = 0; e < 8; ++e) {
                                if (rc + e < n_rows) table[((int64_t)qb * K + c) * nq + qi] = out[e];
                                if (++qi == unq) { qi = 0; ++qb; }
                            }
                        }
                    }
                }
            }
        }
        if (FILTER && pend_key && pend_slot < tiles.cap) pend_dst[pend_slot] = pend_key;
    }

    tc_fence_before();
    __syncthreads();
    if (warp == 0) {
        tc_fence_after();
        tmem_dealloc(tmem, G1_TMEM_COLS);
    }
}

// ------------------------------------------------------------------------------------------------ host side ------
typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                  const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

static EncodeTiledFn encode_fn()
{
    static EncodeTiledFn fn = nullptr;
    if (!fn) {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = (EncodeTiledFn)p;
    }
    return fn;
}

// Digit planes [3][rows][128] int8 as a 3-D tensor (128 bytes, rows, 3 planes); box = (128, box_rows, box_planes);
// rows past the end read as zeros.
int make_plane_map(CUtensorMap *map, const int8_t *planes, int64_t rows, int box_rows, int box_planes)
{
    EncodeTiledFn fn = encode_fn();
    if (!fn) return fail(CHIMERA_CUDA_ERROR, "cuTensorMapEncodeTiled is not available from the driver");
    cuuint64_t dims[3] = {(cuuint64_t)G1_ROW_BYTES, (cuuint64_t)rows, 3};
    cuuint64_t strides[2] = {(cuuint64_t)G1_ROW_BYTES, (cuuint64_t)rows * G1_ROW_BYTES};
    cuuint32_t box[3] = {(cuuint32_t)G1_ROW_BYTES, (cuuint32_t)box_rows, (cuuint32_t)box_planes};
    cuuint32_t estr[3] = {1, 1, 1};
    CUresult r = fn(map, CU_TENSOR_MAP_DATA_TYPE_UINT8, 3, (void *)planes, dims, strides, box, estr,
                    CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                    CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) return fail(CHIMERA_CUDA_ERROR, "cuTensorMapEncodeTiled failed with code %d", (int)r);
    return CHIMERA_OK;
}

// One launch of the kernel over `c_tiles` centroid tiles (see G1Tiles for which).
template <bool FILTER, bool TABLE>
static int launch_g1_tiles(const Index &ix, const Params &p, const CUtensorMap &map_q, int c_tiles, int32_t *table,
                           uint8_t *table8, uint32_t *status, const G1Tiles &tiles, cudaStream_t st)
{
    const int64_t rows = (int64_t)p.B * p.nq;
    const int n_tiles = (int)((rows + G1_N - 1) / G1_N);
    // about eight waves of two CTAs per SM, so the last wave is mostly full; a launch over few centroid tiles (the
    // sample) fills one wave instead, because a CTA's start-up costs as much as three tiles
    // -- unless it will hardly ever have anything to do (redo): then one CTA per centroid tile
    int splits = tiles.redo ? 1 : c_tiles < 2 * ix.sm_count ? (2 * ix.sm_count) / c_tiles : (16 * ix.sm_count + c_tiles - 1) / c_tiles;
    if (splits > n_tiles) splits = n_tiles;
    if (splits < 1) splits = 1;
    const int tiles_per_split = (n_tiles + splits - 1) / splits;
    dim3 grid((unsigned)c_tiles, (unsigned)((n_tiles + tiles_per_split - 1) / tiles_per_split));
    const long long limit = wait_limit_cycles();
    const int skip = fault_skip_tma_loads();
#define CHIMERA_G1_LAUNCH(KS)                                                                                          \
    do {                                                                                                               \
        CHIMERA_CUDA(allow_shared(score_table_umma<KS, FILTER, TABLE>, G1_SMEM));                                      \
        launch(score_table_umma<KS, FILTER, TABLE>, grid, G1_THREADS, G1_SMEM, st, ix.cdig, map_q, ix.K, p.nq, rows, n_tiles,     \
                                                                        tiles_per_split, table, table8, status, limit, \
                                                                        skip, tiles);                                  \
    } while (0)
    switch (ix.D / 32) {                       // MMA steps of 32 dimensions
    case 1: CHIMERA_G1_LAUNCH(1); break;
    case 2: CHIMERA_G1_LAUNCH(2); break;
    case 3: CHIMERA_G1_LAUNCH(3); break;
    default: CHIMERA_G1_LAUNCH(4); break;
    }
#undef CHIMERA_G1_LAUNCH
    CHIMERA_CUDA(cudaGetLastError());
    return CHIMERA_OK;
}

int launch_score_table(const Index &ix, const Params &p, const float *queries, int8_t *qdig, int8_t *qdig4, int32_t *table,
                       uint8_t *table8, uint32_t *status, cudaStream_t st, uint32_t *clear, int64_t clear_n)
{
    const int64_t rows = (int64_t)p.B * p.nq;
    int rc = launch_digits(queries, rows, ix.D, ix.nbits, qdig, true, qdig4, p.nq, status, st, clear, clear_n);
    if (rc) return rc;
    CUtensorMap map_q;
    if ((rc = make_plane_map(&map_q, qdig, table_rows(rows), G1_N, 3))) return rc;        // one load brings a tile's three planes
    const G1Tiles all = {0, 0, nullptr, nullptr, nullptr, 0, nullptr};
    if ((rc = launch_g1_tiles<false, true>(ix, p, map_q, (int)((ix.K + G1_M - 1) / G1_M), table, table8, status, all, st)))
        return rc;
    count_launch(SLOT_G1, 2);
    return CHIMERA_OK;
}

// Stages 1 and 2a together (Sec. 3.2 step 1 on top of Definition 1's products): the table of a sample of the centroid
// tiles first, from it a lower bound per query token on the score of the token's true nprobe-th best centroid, then
// the rest of the table with every score at or above that bound queued beside it (the sample's own scores are queued
// by a scan of their rows), and the nprobe best keys of each queue.  The result is the exact top nprobe by (score
// descending, centroid id ascending): a centroid that belongs to it has a score >= the bound, so it is queued.
// A query with a token whose queue overflowed is redone by the table scan of the separate probe stage.
int launch_score_table_probes(const Index &ix, const Params &p, const Layout &L, const float *queries, int8_t *qdig, int8_t *qdig4,
                              int32_t *table, bool keep_table, uint8_t *table8, char *ws, uint32_t *status, cudaStream_t st,
                              uint32_t *clear, int64_t clear_n)
{
    const int64_t rows = (int64_t)p.B * p.nq;
    int rc = launch_digits(queries, rows, ix.D, ix.nbits, qdig, true, qdig4, p.nq, status, st, clear, clear_n);
    if (rc) return rc;
    CUtensorMap map_q;
    if ((rc = make_plane_map(&map_q, qdig, table_rows(rows), G1_N, 3))) return rc;
    const int c_tiles = (int)((ix.K + G1_M - 1) / G1_M);
    const int stride = L.pq_stride;
    const int n_sample = (c_tiles + stride - 1) / stride;
    int32_t *thr = (int32_t *)(ws + L.pq_thr), *cnt = (int32_t *)(ws + L.pq_cnt);
    unsigned long long *keys = (unsigned long long *)(ws + L.pq_keys);

    const G1Tiles sample = {stride, 1, nullptr, nullptr, nullptr, 0, nullptr};
    if ((rc = launch_g1_tiles<false, true>(ix, p, map_q, n_sample, table, table8, status, sample, st))) return rc;
    if ((rc = launch_probe_sample(ix, p, L, table, ws, n_sample, st))) return rc;
    const G1Tiles rest = {stride, 0, thr, cnt, keys, L.pq_cap, nullptr};
    rc = keep_table ? launch_g1_tiles<true, true>(ix, p, map_q, c_tiles - n_sample, table, table8, status, rest, st)
                    : launch_g1_tiles<true, false>(ix, p, map_q, c_tiles - n_sample, nullptr, nullptr, status, rest, st);
    if (rc) return rc;
    count_launch(SLOT_G1, 3);
    return CHIMERA_OK;
}

// The tiles that launch_score_table_probes left out of the table (keep_table false), for the queries that `redo` flags.
int launch_score_table_redo(const Index &ix, const Params &p, const Layout &L, const int8_t *qdig, int32_t *table,
                            const int32_t *redo, uint32_t *status, cudaStream_t st)
{
    CUtensorMap map_q;
    const int rc = make_plane_map(&map_q, qdig, table_rows((int64_t)p.B * p.nq), G1_N, 3);
    if (rc) return rc;
    const int c_tiles = (int)((ix.K + G1_M - 1) / G1_M);
    const int n_sample = (c_tiles + L.pq_stride - 1) / L.pq_stride;
    const G1Tiles rest = {L.pq_stride, 0, nullptr, nullptr, nullptr, 0, redo};
    return launch_g1_tiles<false, true>(ix, p, map_q, c_tiles - n_sample, table, nullptr, status, rest, st);
}

}  // namespace chimera
