// Stage 3, first cut of a batch: the bounds hi0 of g3_filter.cu for ALL queries of a group in one pass over the corpus.
//
// The scan of g3_filter.cu takes one query at a time, so a token is looked up once for each query that has its document as a
// candidate.  Here e(c) of up to 256 queries stands side by side in one row of codes, a token's row is read once and its codes
// are added up for all of them: documents that are not candidates of a query are summed in vain, and a row costs one line of
// the load pipe whatever it holds.  That pays as soon as the queries' candidates hold a few times the corpus's tokens
// (batch_scan_used).
//
// A code is ceil(e / step) with a step per query, chosen from a sample so that few centroids reach past the largest code (the
// ones near a query token).  What those have above it is added to the documents of their posting lists afterwards.  The lists
// name a document once, which is all a bound needs: a centroid's second token in a document cannot raise a maximum.
// Codes have 6 bits and a byte each, so that four add up without a carry.  (Half a byte, 4 bits: 730 instead of 885 us for the
// scan of Mid's batch of 256, but four times the step: a third more candidates kept, or long lists to add.)
//
//   batch_quantum_kernel   step and sum of theta of each query
//   batch_excess_kernel    the codes, and the list of centroids with more than BS_TOP steps (from the 8-bit
//                          table; batch_excess_exact_kernel for other query lengths)
//   batch_scan_kernel      hi0 of every candidate
//   batch_over_kernel      the rest of the listed centroids
//   batch_hist_kernel      histogram of the bounds, for the choice of the seeds
#include "g3_filter.cuh"

namespace chimera {

constexpr int BS_TILE = 64;               // documents per tile
constexpr int BS_THREADS = 256;
constexpr int BS_OVER = CHIMERA_LISTED_ROOM;     // listed centroids per query; with more of them all rows are looked at again

constexpr int BS_TOP = 63;                // the largest code
constexpr int BS_MAX_LEN = 65535 / BS_TOP;              // tokens of a document: sums are 16-bit fields

// Queries side by side in a row, a byte each.
int batch_group(const Params &p)
{
    return p.B <= 8 ? 8 : p.B <= 16 ? 16 : p.B <= 32 ? 32 : p.B <= 64 ? 64 : p.B <= 128 ? 128 : 256;
}
static int batch_groups(const Params &p) { return (p.B + batch_group(p) - 1) / batch_group(p); }

// When a batch is scanned this way: by the SM cycles of both forms.  Cycles a token and SM by the bytes of a row, measured on
// 200,000 to 500,000 documents: 8 bytes 0.95, 16 1.2, 32 1.3, 64 1.4, 128 2.4, 256 4.3 (a line of the load pipe, then what L2
// delivers).  The scan by query takes 4.3 tokens a cycle from 16-bit values and 2.2 from 6-bit codes, of the candidates only.  The
// table has to stay in L2 beside what streams past: 32 of its 126 MB.  Query lengths other than 32 and 64 have no 8-bit table when the
// step is chosen, and pay 10 to 20 us for its rows: 3 million token cycles (224 calls on 8,000 to 150,000 documents, both forms: without
// that, 21 tokens lost up to 10 % of a call and 106 up to 9 %; with it nothing loses more than 1 %).
bool batch_scan_used(const Index &ix, const Params &p)
{
    if (!filter_used(ix, p) || ix.max_doclen > BS_MAX_LEN) return false;
    const int row = batch_group(p);
    if ((int64_t)row * ix.K > (32LL << 20)) return false;
    const double cycles = row == 8 ? 0.95 : row == 16 ? 1.2 : row == 32 ? 1.3 : row == 64 ? 1.4 : row == 128 ? 2.4 : 4.3;
    const double fixed = coarse_supported(p.nq) ? 0.0 : 3e6;
    return batch_groups(p) * (double)ix.T * cycles + fixed < (double)p.B * expected_tokens(ix, p) / (ix.K <= 106496 ? 4.3 : 2.2);
}
size_t batch_table_bytes(const Index &ix, const Params &p)
{
    return (size_t)batch_groups(p) * (size_t)(ix.K + 1) * (size_t)batch_group(p);
}
// Per query: step and base, the listed centroids and their number.
size_t batch_over_bytes(const Params &p) { return (size_t)p.B * (sizeof(int2) * (1 + BS_OVER) + sizeof(int32_t)); }
struct BatchScratch { int2 *scale, *over; int32_t *n_over; };
static BatchScratch batch_scratch(const Params &p, const Layout &L, char *ws)
{
    BatchScratch s;
    s.scale = (int2 *)(ws + L.flt_over);
    s.over = s.scale + p.B;
    s.n_over = (int32_t *)(s.over + (size_t)p.B * BS_OVER);
    return s;
}

// Code k of the four in a word: even codes in bytes 0 and 1, odd ones in bytes 2 and 3, so that a mask leaves two neighbours in
// 16-bit fields.
__device__ __forceinline__ int code_shift(int k) { return 16 * (k & 1) + 8 * (k >> 1); }
// ceil(e / step) by a multiplication: e + step - 1 < 2^17 and floor(2^32 / step) + 1 is exact for numerators up to 2^32 / step.
__device__ __forceinline__ uint32_t step_inverse(uint32_t step) { return step > 1 ? 0xffffffffu / step + 1u : 0u; }
__device__ __forceinline__ uint32_t code_of(uint32_t e, uint32_t step, uint32_t inv)
{
    return step > 1 ? __umulhi(e + step - 1u, inv) : e;
}
__device__ __forceinline__ void list_over(int32_t *n_over, int2 *over, int b, int64_t c, uint32_t rest)
{
    const int at = atomicAdd(&n_over[b], 1);
    if (at < BS_OVER) over[(int64_t)b * BS_OVER + at] = make_int2((int)c, (int)rest);
}

// e(c) of a row of the exact table, on all lanes of a warp (lane = column), in units of 2^us, rounded up.  (A score that reaches
// theta counts, so that zero means a centroid with none.)
__device__ __forceinline__ uint32_t exact_row_excess(const int32_t *row, int nq, const int32_t *th, int us, int lane)
{
    int e = 0;
    for (int w = lane; w < nq; w += 32) e += max(__ldg(row + w) - ((th[w] << 16) - 1), 0);
    return ((uint32_t)__reduce_add_sync(0xffffffffu, e) + ((1u << us) - 1)) >> us;       // (127 columns: below 2^31)
}

// grid (B).  The smallest cap that at most `rank` of the m sampled rows (every step-th one) exceed; BS_TOP of the query's steps
// reach it.  WORDS: words of an 8-bit row (q_len 32 / 64), or 0: from the exact table.
template <int WORDS>
__global__ void __launch_bounds__(SEL_THREADS)
batch_quantum_kernel(const int32_t *__restrict__ table, const uint8_t *__restrict__ table8, int64_t K, int nq,
                     const int32_t *__restrict__ theta, int m, int step, int rank, int us, int2 *__restrict__ scale,
                     int32_t *__restrict__ n_over)
{
    pdl_entry();
    constexpr int W = WORDS > 0 ? WORDS : 1;
    __shared__ int hist[SEL_THREADS];                        // of e in units of 2^16, the last bin open
    __shared__ int warp_part[32];
    __shared__ uint2 tm1[W];
    __shared__ int s_sum, s_bin;
    __shared__ int32_t s_th[128];
    const int b = blockIdx.x, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int32_t *th = theta + (int64_t)b * nq;
    hist[threadIdx.x] = 0;
    if (threadIdx.x < nq) s_th[threadIdx.x] = th[threadIdx.x];
    if (threadIdx.x == 0) s_bin = 0;
    __syncthreads();
    if (threadIdx.x < 4 * W && (threadIdx.x & 3) == 0 && WORDS > 0) {
        const int32_t *t = s_th + threadIdx.x;
        tm1[threadIdx.x >> 2] = make_uint2((uint32_t)(t[0] - 1) | (uint32_t)(t[2] - 1) << 16,
                                           (uint32_t)(t[1] - 1) | (uint32_t)(t[3] - 1) << 16);
    }
    if (warp == 0) {
        int s = 0;
        for (int i = lane; i < nq; i += 32) s += s_th[i];
        s = __reduce_add_sync(0xffffffffu, s);
        if (lane == 0) s_sum = s;
    }
    __syncthreads();
    if constexpr (WORDS > 0) {
        const uint4 *tb = reinterpret_cast<const uint4 *>(table8 + (int64_t)b * K * 4 * WORDS);
#pragma unroll 4
        for (int r = threadIdx.x; r < m; r += SEL_THREADS) {
            const int e = filter_row_excess<W>(tb + (int64_t)r * step * (W / 4), tm1, s_sum - nq);
            atomicAdd(&hist[e < SEL_THREADS ? e : SEL_THREADS - 1], 1);
        }
    } else {
        const int32_t *tb = table + (int64_t)b * K * nq;
        for (int r0 = warp; r0 < m; r0 += 8 * 32) {          // eight rows in flight
            int v[8][4], e[8];
#pragma unroll
            for (int u = 0; u < 8; ++u)
#pragma unroll
                for (int w = 0; w < 4; ++w)
                    v[u][w] = r0 + 32 * u < m && lane + 32 * w < nq ? __ldg(tb + (int64_t)(r0 + 32 * u) * step * nq + lane + 32 * w) : 0;
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                e[u] = 0;
#pragma unroll
                for (int w = 0; w < 4; ++w) e[u] += max(v[u][w] - (lane + 32 * w < nq ? (s_th[lane + 32 * w] << 16) - 1 : 0), 0);
                e[u] = __reduce_add_sync(0xffffffffu, e[u]) >> 16;
                if (lane == 0 && r0 + 32 * u < m) atomicAdd(&hist[e[u] < SEL_THREADS ? e[u] : SEL_THREADS - 1], 1);
            }
        }
    }
    __syncthreads();
    const int bin = SEL_THREADS - 1 - (int)threadIdx.x, mine = hist[bin];
    int total;
    const int above = sel_block_scan(mine, &total, warp_part);
    if (above <= rank && rank < above + mine) s_bin = bin;
    __syncthreads();
    if (threadIdx.x == 0) {
        const int cap = ((s_bin + 1) << (16 - us)) - 1, q = (cap + BS_TOP - 1) / BS_TOP;
        scale[b] = make_int2(s_sum << (16 - us), q > 1 ? q : 1);
        n_over[b] = 0;
    }
}

// grid (blocks, words of all rows / CW).  Codes of four queries to a word and CW words at a time, a thread per centroid and word:
// a stream of the 8-bit table (Mid, batch 256: 537 MB), a warp's 32 rows of a query side by side; the words change places in
// shared memory so that a row's CW are stored together.  Row K stays zero: the scan sends positions behind a document's
// end there.
template <int WORDS, int CW>
__global__ void __launch_bounds__(BS_THREADS)
batch_excess_kernel(const uint8_t *__restrict__ table8, int64_t K, int B, int group, const int32_t *__restrict__ theta,
                    const int2 *__restrict__ scale, uint32_t *__restrict__ out, int32_t *__restrict__ n_over,
                    int2 *__restrict__ over, uint32_t *__restrict__ mask, FirstCut cut)
{
    pdl_entry();
    constexpr int NQ = 4 * WORDS, ROWS = BS_THREADS / CW, QB = 4 * CW;
    __shared__ uint2 tm1[QB][WORDS];
    __shared__ int s_sum[QB];
    __shared__ uint32_t s_step[QB], s_inv[QB];
    __shared__ uint32_t s_word[2][ROWS][CW + 1];
    const int row_words = group / 4, b0 = (int)blockIdx.y * QB;
    if (!cut.on()) return;
    for (int i = threadIdx.x; i < QB * WORDS; i += BS_THREADS) {
        const int b = b0 + i / WORDS;
        uint2 v = make_uint2(0x00ff00ffu, 0x00ff00ffu);
        if (b < B) {
            const int4 t = __ldg(reinterpret_cast<const int4 *>(theta + (int64_t)b * NQ) + i % WORDS);
            v = make_uint2((uint32_t)(t.x - 1) | (uint32_t)(t.z - 1) << 16, (uint32_t)(t.y - 1) | (uint32_t)(t.w - 1) << 16);
        }
        tm1[i / WORDS][i % WORDS] = v;
    }
    if (threadIdx.x < QB) {
        const int b = b0 + threadIdx.x;
        const int2 s = b < B ? scale[b] : make_int2(0, 1);
        s_sum[threadIdx.x] = s.x - NQ;                       // (us is 16: the sum of theta itself)
        s_step[threadIdx.x] = (uint32_t)s.y;
        s_inv[threadIdx.x] = step_inverse((uint32_t)s.y);
    }
    __syncthreads();
    const int word = threadIdx.x / ROWS, row = threadIdx.x % ROWS, q0 = 4 * word, first = b0 + q0;
    // (a block's queries are of one group)
    uint32_t *dst = out + (size_t)(b0 / group) * (size_t)(K + 1) * row_words + b0 % group / 4;
    int buf = 0;
    for (int64_t c0 = (int64_t)blockIdx.x * ROWS; c0 <= K; c0 += (int64_t)gridDim.x * ROWS, buf ^= 1) {
        const int64_t c = c0 + row;
        uint32_t packed = 0;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int b = first + k;
            if (b >= B) break;                               // (the same for all lanes)
            uint32_t e = 0;
            if (c < K) {
                const uint4 *src = reinterpret_cast<const uint4 *>(table8 + ((int64_t)b * K + c) * NQ);
                e = (uint32_t)filter_row_excess<WORDS>(src, tm1[q0 + k], s_sum[q0 + k]);
            }
            const uint32_t near = __ballot_sync(0xffffffffu, e > 0);
            if ((threadIdx.x & 31) == 0 && c < K) mask[(int64_t)b * ((K + 31) / 32) + (c >> 5)] = near;
            const uint32_t step = s_step[q0 + k];
            uint32_t code = code_of(e, step, s_inv[q0 + k]);
            if (code > BS_TOP) {
                code = BS_TOP;
                list_over(n_over, over, b, c, e - BS_TOP * step);
            }
            packed |= code << code_shift(k);
        }
        s_word[buf][row][word] = packed;
        __syncthreads();                                     // (the other buffer's readers are past the barrier before)
        const int64_t cw = c0 + threadIdx.x / CW;
        if (cw <= K) dst[cw * row_words + threadIdx.x % CW] = s_word[buf][threadIdx.x / CW][threadIdx.x % CW];
    }
}

// The same from the exact table, for any q_len: a warp per query, eight centroids at a time, and the 8-bit rows that the
// second bound looks up on the way (as filter_excess_exact_kernel makes them).  grid (blocks, queries of all rows / 8).
template <int NQW>
__global__ void __launch_bounds__(BS_THREADS)
batch_excess_exact_kernel(const int32_t *__restrict__ table, int64_t K, int nq, int B, int group, const int32_t *__restrict__ theta,
                          int us, const int2 *__restrict__ scale, uint8_t *__restrict__ table8, uint32_t *__restrict__ out,
                          int32_t *__restrict__ n_over, int2 *__restrict__ over, uint8_t *__restrict__ mask)
{
    pdl_entry();
    constexpr int PER = 8, pitch8 = 32 * NQW;
    __shared__ uint8_t s_code[2][PER][8];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int first = (int)blockIdx.y * 8, b = first + warp, row_words = group / 4, g = first / group;
    const bool live = b < B;
    uint32_t *dst = out + (size_t)g * (size_t)(K + 1) * row_words + (first - g * group) / 4;
    const int64_t row0 = live ? (int64_t)b * K : 0;
    const int32_t *tb = table + row0 * nq;
    uint8_t *t8 = table8 + row0 * pitch8;
    int th[NQW];
#pragma unroll
    for (int w = 0; w < NQW; ++w) th[w] = live && lane + 32 * w < nq ? (theta[(int64_t)b * nq + lane + 32 * w] << 16) - 1 : 0;
    const uint32_t step = live ? (uint32_t)scale[b].y : 1u, inv = step_inverse(step);
    const int64_t groups = (K + 1 + PER - 1) / PER;
    int buf = 0;
    for (int64_t gr = blockIdx.x; gr < groups; gr += gridDim.x, buf ^= 1) {
        int e[PER];
        uint32_t coarse[PER];
#pragma unroll
        for (int r = 0; r < PER; ++r) { e[r] = 0; coarse[r] = 0u; }
#pragma unroll
        for (int w = 0; w < NQW; ++w) {
            int v[PER];
#pragma unroll
            for (int r = 0; r < PER; ++r)
                v[r] = (live && lane + 32 * w < nq && gr * PER + r < K) ? __ldg(tb + (gr * PER + r) * nq + lane + 32 * w) : 0;
#pragma unroll
            for (int r = 0; r < PER; ++r) {
                coarse[r] |= (uint32_t)__vimin_s32_relu(v[r] >> 16, 255) << (8 * w);
                e[r] += max(v[r] - th[w], 0);         // (a column or row past the end has no value above its threshold)
            }
        }
        if (live)
#pragma unroll
            for (int r = 0; r < PER; ++r) {
                if (gr * PER + r >= K) break;
                uint8_t *row = t8 + (gr * PER + r) * pitch8;
                if constexpr (NQW == 1) row[lane] = (uint8_t)coarse[r];
                else if constexpr (NQW == 2) reinterpret_cast<uint16_t *>(row)[lane] = (uint16_t)coarse[r];
                else reinterpret_cast<uint32_t *>(row)[lane] = coarse[r];
            }
        uint32_t mine = 0, near = 0;
#pragma unroll
        for (int r = 0; r < PER; ++r) {
            // the sum of 127 columns stays below 2^31; + the rounding, so add in unsigned
            const uint32_t s = ((uint32_t)__reduce_add_sync(0xffffffffu, e[r]) + ((1u << us) - 1)) >> us;
            near |= (uint32_t)(s > 0) << r;
            if (lane == r) mine = s;
        }
        if (NQW > 1 && live && lane == 0 && gr * PER < K) mask[(int64_t)b * ((K + 31) / 32) * 4 + gr] = (uint8_t)near;
        if (lane < PER) {
            uint32_t code = code_of(mine, step, inv);
            if (code > BS_TOP) {
                code = BS_TOP;
                list_over(n_over, over, b, gr * PER + lane, mine - BS_TOP * step);
            }
            s_code[buf][lane][warp] = (uint8_t)code;
        }
        __syncthreads();                                 // (the other buffer's readers are past the barrier before)
        if (threadIdx.x < 2 * PER && gr * PER + threadIdx.x / 2 <= K) {
            const int r = threadIdx.x / 2, w = threadIdx.x % 2;
            uint32_t packed = 0;
#pragma unroll
            for (int k = 0; k < 4; ++k) packed |= (uint32_t)s_code[buf][r][4 * w + k] << code_shift(k);
            dst[(gr * PER + r) * row_words + w] = packed;
        }
    }
}

// x * one + a with `one` = 1 that the compiler does not know: an addition on the multiply-add pipe (the masks and shifts below
// keep the integer pipe busy, which takes an instruction every other cycle).
__device__ __forceinline__ uint32_t mad_one(uint32_t x, uint32_t one, uint32_t a)
{
    uint32_t r;
    asm("mad.lo.u32 %0, %1, %2, %3;" : "=r"(r) : "r"(x), "r"(one), "r"(a));
    return r;
}

// grid (blocks, groups).  A block takes tiles of 64 documents; a warp DPW of them at a time, 32 / DPW lanes each, LPR lanes of
// WPL words to a row, so a load of the warp reads 32 / LPR tokens; U such loads are in flight and the ids of the next ones
// behind them.  Codes are added as bytes, four tokens at a time, then as 16-bit fields; the token groups of a document
// are folded with shuffles.  The sums wait in shared memory until the tile is done, and then go to the candidates among its
// documents: ranks[query][word] = 32 documents' candidate bits and the number of candidates before them.
// Where documents share a warp they are taken by length: there is less to fold, and one document's end costs a part of the warp.
template <int LPR, int WPL, int DPW, int U>
__global__ void __launch_bounds__(BS_THREADS, LPR >= 4 ? 3 : 4)
batch_scan_kernel(const uint32_t *__restrict__ tab, int64_t K, const int32_t *__restrict__ cids,
                  const int64_t *__restrict__ doc_off, int64_t N, int n_tiles, const uint2 *__restrict__ ranks, int64_t words,
                  const int2 *__restrict__ scale, int B, int64_t maxc, int32_t *__restrict__ hi0, uint32_t one, FirstCut cut)
{
    pdl_entry();
    constexpr int ROW = LPR * WPL, GQ = 4 * ROW;           // words of a row, queries of a group
    constexpr int LPD = 32 / DPW, TG = LPD / LPR;            // lanes and token groups of a document
    constexpr int NR = 2 * WPL;                              // 16-bit pairs of a lane
    constexpr int STRIDE = GQ + 8;
    constexpr int TPI = U * TG, IDS = (TPI + LPD - 1) / LPD; // tokens of a document per iteration, their ids per lane
    constexpr int ROUNDS = BS_TILE / (8 * DPW);
    constexpr int DPT = BS_TILE * GQ / BS_THREADS;           // documents per thread when the sums are handed out
    constexpr int RK = DPT > 32 ? 2 : 1;
    __shared__ __align__(16) uint16_t s_acc[BS_TILE * STRIDE];
    __shared__ int s_t0[2][BS_TILE], s_len[2][BS_TILE];
    __shared__ uint8_t s_ord[2][BS_TILE];
    if (!cut.on()) return;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int dl = lane % LPD, dg = lane / LPD, grp = dl / LPR, sub = lane % LPR;
    const int b0 = blockIdx.y * GQ;
    const uint32_t *tb = tab + (size_t)blockIdx.y * (size_t)(K + 1) * ROW + sub * WPL;
    const int q = tid % GQ, part = tid / GQ;                 // the query and documents [part DPT, + DPT) that this thread hands out
    const bool hands = b0 + q < B;
    const int2 sc = hands ? scale[b0 + q] : make_int2(0, 0);
    int32_t *out = hi0 + (int64_t)(b0 + q) * maxc;
    auto range = [&](int tile, int &t0, int &len) {
        const int64_t d = (int64_t)tile * BS_TILE + tid;
        t0 = len = 0;
        if (tid < BS_TILE && tile < n_tiles && d < N) {
            const int64_t a = doc_off[d];
            t0 = (int)a;
            len = (int)(doc_off[d + 1] - a);
        }
    };
    auto order = [&](int buf) {                              // longest first
        if (DPW > 1 && tid < BS_TILE) {
            const int mine = s_len[buf][tid] << 6 | tid;
            int rank = 0;
#pragma unroll 16
            for (int i = 0; i < BS_TILE; ++i) rank += (s_len[buf][i] << 6 | i) > mine ? 1 : 0;
            s_ord[buf][rank] = (uint8_t)tid;
        }
    };
    int buf = 0;
    if ((int)blockIdx.x < n_tiles) {
        int t0, len;
        range(blockIdx.x, t0, len);
        if (tid < BS_TILE) { s_t0[0][tid] = t0; s_len[0][tid] = len; }
    }
    __syncthreads();
    order(0);
    if (DPW > 1) __syncthreads();
    for (int tile = blockIdx.x; tile < n_tiles; tile += gridDim.x, buf ^= 1) {
        int nx_t0, nx_len;
        range(tile + (int)gridDim.x, nx_t0, nx_len);
        uint2 rk[RK];
#pragma unroll
        for (int w = 0; w < RK; ++w) {
            const int64_t word = (int64_t)tile * (BS_TILE / 32) + part * DPT / 32 + w;
            rk[w] = hands && word < words ? __ldg(ranks + (int64_t)(b0 + q) * words + word) : make_uint2(0u, 0u);
        }
        // documents in rounds of 8 DPW; every other round hands them to the warps in reverse, so that all get as much
        auto doc_of = [&](int r) {
            if (DPW == 1) return 8 * r + warp;
            return (int)s_ord[buf][((r & 1) ? 8 * (r + 1) - 1 - warp : 8 * r + warp) * DPW + dg];
        };
        int32_t id[IDS];
        auto load_ids = [&](int t0, int from, int len) {
#pragma unroll
            for (int k = 0; k < IDS; ++k) {
                const int i = from + LPD * k + dl;
                id[k] = i < len ? DBG_CID(__ldg(cids + DBG_TOK((int64_t)t0 + i))) : (int32_t)K;
            }
        };
        int d = doc_of(0), t0 = s_t0[buf][d], len = s_len[buf][d];
        load_ids(t0, 0, len);
        for (int r = 0; r < ROUNDS; ++r) {
            const int dn = r + 1 < ROUNDS ? doc_of(r + 1) : d;
            const int t0n = s_t0[buf][dn], lenn = s_len[buf][dn];
            const int most = DPW > 1 ? __reduce_max_sync(0xffffffffu, len) : len;
            uint32_t sum[NR];
#pragma unroll
            for (int x = 0; x < NR; ++x) sum[x] = 0u;
            int base = 0;
            do {
                uint32_t v[U][WPL];
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const int32_t c = LPR == 1 && DPW == 1 ? id[u] : __shfl_sync(0xffffffffu, id[u * TG / LPD], u * TG % LPD + grp, LPD);
                    const uint32_t *src = tb + (uint64_t)(uint32_t)c * ROW;
                    if constexpr (WPL == 4) {
                        const uint4 x = __ldg(reinterpret_cast<const uint4 *>(src));
                        v[u][0] = x.x; v[u][1] = x.y; v[u][2] = x.z; v[u][3] = x.w;
                    } else {
                        const uint2 x = __ldg(reinterpret_cast<const uint2 *>(src));
                        v[u][0] = x.x; v[u][1] = x.y;
                    }
                }
                base += TPI;
                const bool more = base < most;
                load_ids(more ? t0 : t0n, more ? base : 0, more ? len : r + 1 < ROUNDS ? lenn : 0);
#pragma unroll
                for (int u = 0; u < U; u += 4)
#pragma unroll
                    for (int w = 0; w < WPL; ++w) {          // 4 times 63 fit a byte
                        const uint32_t s = v[u][w] + v[u + 1][w] + v[u + 2][w] + v[u + 3][w];
                        sum[2 * w] = mad_one(s & 0x00ff00ffu, one, sum[2 * w]);
                        sum[2 * w + 1] = mad_one((s >> 8) & 0x00ff00ffu, one, sum[2 * w + 1]);
                    }
            } while (base < most);
            // fold the token groups: an exchange keeps one half of the registers while there are several
            int nreg = NR, start = 0;
            uint32_t dup = 0;
#pragma unroll
            for (int o = LPD / 2; o >= LPR; o >>= 1) {
                if (nreg > 1) {
                    const int half = nreg >> 1;
                    const bool up = (lane & o) != 0;
#pragma unroll
                    for (int x = 0; x < NR / 2; ++x)
                        if (x < half) {
                            const uint32_t send = up ? sum[x] : sum[x + half], keep = up ? sum[x + half] : sum[x];
                            sum[x] = keep + __shfl_xor_sync(0xffffffffu, send, o);
                        }
                    start += up ? half : 0;
                    nreg = half;
                } else {
                    sum[0] += __shfl_xor_sync(0xffffffffu, sum[0], o);
                    dup |= (uint32_t)o;
                }
            }
            if ((lane & dup) == 0) {
                uint16_t *dst = s_acc + d * STRIDE + sub * WPL * 4 + 2 * start;
                if (nreg >= 4) {
#pragma unroll
                    for (int x = 0; x < NR; x += 4)
                        if (x < nreg) *reinterpret_cast<uint4 *>(dst + 2 * x) = make_uint4(sum[x], sum[x + 1], sum[x + 2], sum[x + 3]);
                } else if (nreg == 2) *reinterpret_cast<uint2 *>(dst) = make_uint2(sum[0], sum[1]);
                else *reinterpret_cast<uint32_t *>(dst) = sum[0];
            }
            d = dn; t0 = t0n; len = lenn;
        }
        if (tid < BS_TILE) { s_t0[buf ^ 1][tid] = nx_t0; s_len[buf ^ 1][tid] = nx_len; }
        __syncthreads();
        order(buf ^ 1);
        if (hands) {
#pragma unroll
            for (int w = 0; w < RK; ++w) {
                const int s = part * DPT & 31, doc0 = (part * DPT & ~31) + 32 * w;
                uint32_t bits = DPT >= 32 ? rk[w].x : rk[w].x & (((1u << (DPT & 31)) - 1u) << s);
                int64_t pos = (int64_t)rk[w].y + __popc(rk[w].x & ((1u << s) - 1u));
                while (bits) {
                    const int i = __ffs(bits) - 1;
                    bits &= bits - 1;
                    if (pos < maxc) out[pos] = sc.x + sc.y * (int)s_acc[(doc0 + i) * STRIDE + q];
                    ++pos;
                }
            }
        }
        __syncthreads();
    }
}

// grid (blocks, B).  What the listed centroids have above BS_TOP steps, to the candidates in their posting lists; a block per
// centroid.  A query that lists more than there is room for looks at all of its rows again.
template <int WORDS>
__global__ void __launch_bounds__(BS_THREADS)
batch_over_kernel(const int32_t *__restrict__ table, const uint8_t *__restrict__ table8, int64_t K, int nq,
                  const int32_t *__restrict__ theta, int us, const int2 *__restrict__ scale, const int32_t *__restrict__ n_over,
                  const int2 *__restrict__ over, const int64_t *__restrict__ ivf_off, const int32_t *__restrict__ ivf_doc,
                  const uint2 *__restrict__ ranks, int64_t words, int64_t maxc, int32_t *__restrict__ hi0, FirstCut cut)
{
    pdl_entry();
    constexpr int W = WORDS > 0 ? WORDS : 1;
    __shared__ uint2 tm1[W];
    const int b = blockIdx.y, lane = threadIdx.x & 31;
    const bool on = cut.on();
    const int n = n_over[b];
    if (!on) return;
    const uint2 *rb = ranks + (int64_t)b * words;
    int32_t *out = hi0 + (int64_t)b * maxc;
    // entries first, first + stride, ... of a list
    auto add = [&](int64_t c, int rest, int first, int stride) {
        const int64_t end = ivf_off[c + 1];
        for (int64_t e0 = ivf_off[c] + first; e0 < end; e0 += 4 * stride) {
            int32_t d[4];
            uint2 rk[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                d[u] = e0 + u * stride < end ? __ldg(ivf_doc + e0 + u * stride) : -1;
                if (d[u] >= 0 && !DBG_DOC_OK(d[u])) d[u] = -1;
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) rk[u] = d[u] >= 0 ? __ldg(rb + (d[u] >> 5)) : make_uint2(0u, 0u);
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int bit = d[u] & 31;
                if (!(rk[u].x >> bit & 1u)) continue;
                const int64_t pos = (int64_t)rk[u].y + __popc(rk[u].x & ((1u << bit) - 1u));
                if (pos < maxc) atomicAdd(out + pos, rest);
            }
        }
    };
    if (n <= BS_OVER) {
        for (int i = blockIdx.x; i < n; i += gridDim.x) {
            const int2 o = over[(int64_t)b * BS_OVER + i];
            add(o.x, o.y, threadIdx.x, BS_THREADS);
        }
        return;
    }
    const int cap = BS_TOP * scale[b].y, warp = blockIdx.x * 8 + (threadIdx.x >> 5), warps = gridDim.x * 8;
    const int32_t *th = theta + (int64_t)b * nq;
    if constexpr (WORDS > 0) {
        if (threadIdx.x < WORDS) {
            const int32_t *t = th + 4 * threadIdx.x;
            tm1[threadIdx.x] = make_uint2((uint32_t)(t[0] - 1) | (uint32_t)(t[2] - 1) << 16,
                                          (uint32_t)(t[1] - 1) | (uint32_t)(t[3] - 1) << 16);
        }
        __syncthreads();
        const int sum = scale[b].x - nq;
        const uint4 *tb = reinterpret_cast<const uint4 *>(table8 + (int64_t)b * K * 4 * WORDS);
        for (int64_t base = 32LL * warp; base < K; base += 32LL * warps) {
            const int64_t c = base + lane;
            const int e = c < K ? filter_row_excess<W>(tb + c * (W / 4), tm1, sum) : 0;
            unsigned mask = __ballot_sync(0xffffffffu, e > cap);
            for (; mask; mask &= mask - 1) {
                const int l = __ffs(mask) - 1;
                add(base + l, __shfl_sync(0xffffffffu, e, l) - cap, lane, 32);
            }
        }
    } else {
        const int32_t *tb = table + (int64_t)b * K * nq;
        for (int64_t c = warp; c < K; c += warps) {
            const int e = (int)exact_row_excess(tb + c * nq, nq, th, us, lane);
            if (e > cap) add(c, e - cap, lane, 32);
        }
    }
}

// grid (blocks, B): hist[b] (cleared before) of hi0 less the sum of theta.
__global__ void __launch_bounds__(SEL_THREADS)
batch_hist_kernel(const int32_t *__restrict__ hi0, const int32_t *__restrict__ n_cand, int64_t maxc, const int2 *__restrict__ scale,
                  int us, int32_t *__restrict__ hist, FirstCut cut)
{
    pdl_entry();
    __shared__ int s_hist[FILTER_BINS];
    const int b = blockIdx.y;
    const bool on = cut.on();
    const int n = n_cand[b], base = scale[b].x;
    if (!on) return;
    for (int i = threadIdx.x; i < FILTER_BINS; i += SEL_THREADS) s_hist[i] = 0;
    __syncthreads();
    const int32_t *in = hi0 + (int64_t)b * maxc;
    const int64_t stride = gridDim.x * SEL_THREADS;
    for (int64_t j = blockIdx.x * SEL_THREADS + threadIdx.x; j < n; j += 8 * stride) {
        int32_t v[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) v[u] = j + u * stride < n ? in[j + u * stride] : -1;
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const int bin = (v[u] - base) >> (17 - us);
            if (v[u] >= 0) atomicAdd(&s_hist[bin < FILTER_BINS ? bin : FILTER_BINS - 1], 1);
        }
    }
    __syncthreads();
    for (int i = threadIdx.x; i < FILTER_BINS; i += SEL_THREADS)
        if (s_hist[i]) atomicAdd(&hist[(int64_t)b * FILTER_BINS + i], s_hist[i]);
}

// ------------------------------------------------------------------------------------------------ launchers -------
int launch_batch_quantum(const Index &ix, const Params &p, const Layout &L, const int32_t *table, const uint8_t *table8,
                         int us, char *ws, cudaStream_t st)
{
    const BatchScratch s = batch_scratch(p, L, ws);
    const int32_t *theta = (const int32_t *)(ws + L.flt_theta);
    // Centroids aimed at, at most: the query tokens' own (whose e is far above the others') and five times as many more.
    const int64_t wanted = 6 * p.nq < ix.K / 16 ? 6 * p.nq : ix.K / 16;
    const int step = (int)(ix.K / 2048 > 1 ? ix.K / 2048 : 1), m = (int)((ix.K + step - 1) / step);
    const int rank = (int)(wanted * m / ix.K);
    launch(!coarse_supported(p.nq) ? batch_quantum_kernel<0> : p.nq == 32 ? batch_quantum_kernel<8> : batch_quantum_kernel<16>,
           dim3((unsigned)p.B), SEL_THREADS, 0, st, table, table8, ix.K, p.nq, theta, m, step, rank, us, s.scale,
           s.n_over);
    CHIMERA_CUDA(cudaGetLastError());
    count_launch(SLOT_CI);
    return CHIMERA_OK;
}

template <int LPR, int WPL, int DPW, int U>
static void launch_scan(const Index &ix, const Params &p, const uint32_t *tab, const uint2 *ranks, int64_t words, const int2 *scale,
                        int32_t *hi0, FirstCut cut, cudaStream_t st)
{
    const int tiles = (int)((ix.N + BS_TILE - 1) / BS_TILE);
    int64_t gx = (int64_t)ix.sm_count * (LPR >= 4 ? 3 : 4) * 4;      // four waves of resident blocks even out the tiles
    if (gx > tiles) gx = tiles;
    launch(batch_scan_kernel<LPR, WPL, DPW, U>, dim3((unsigned)gx, (unsigned)batch_groups(p)), BS_THREADS, 0, st, tab, ix.K, ix.cids,
           ix.doc_off, ix.N, tiles, ranks, words, scale, p.B, p.maxc, hi0, 1u, cut);
}
template <int WORDS, int CW>
static void launch_excess(const Index &ix, const Params &p, const uint8_t *table8, const int32_t *theta, const BatchScratch &s,
                          uint32_t *tab, uint32_t *mask, FirstCut cut, cudaStream_t st)
{
    const int gy = batch_groups(p) * batch_group(p) / 4 / CW, rows = BS_THREADS / CW;
    int64_t gx = (8LL * ix.sm_count + gy - 1) / gy;
    if (gx > (ix.K + rows) / rows) gx = (ix.K + rows) / rows;
    launch(batch_excess_kernel<WORDS, CW>, dim3((unsigned)gx, (unsigned)gy), BS_THREADS, 0, st, table8, ix.K, p.B, batch_group(p), theta,
           s.scale, tab, s.n_over, s.over, mask, cut);
}
template <int WORDS>
static void launch_excess(const Index &ix, const Params &p, const uint8_t *table8, const int32_t *theta, const BatchScratch &s,
                          uint32_t *tab, uint32_t *mask, FirstCut cut, cudaStream_t st)
{
    const int group = batch_group(p);
    if (group == 8) launch_excess<WORDS, 2>(ix, p, table8, theta, s, tab, mask, cut, st);
    else if (group == 16) launch_excess<WORDS, 4>(ix, p, table8, theta, s, tab, mask, cut, st);
    else launch_excess<WORDS, 8>(ix, p, table8, theta, s, tab, mask, cut, st);
}

int launch_batch_scan(const Index &ix, const Params &p, const Layout &L, const int32_t *table, uint8_t *table8, int us,
                      const int32_t *n_cand, int32_t *hi0, char *ws, cudaStream_t st)
{
    const BatchScratch s = batch_scratch(p, L, ws);
    const int32_t *theta = (const int32_t *)(ws + L.flt_theta);
    const FirstCut cut = first_cut(p, L, ws);
    const uint2 *ranks = (const uint2 *)(ws + L.ranks);
    uint32_t *tab = (uint32_t *)(ws + L.flt_tab), *mask = (uint32_t *)(ws + L.flt_mask);
    const int group = batch_group(p);
    const bool wide = coarse_supported(p.nq);
    if (p.nq == 32) {
        launch_excess<8>(ix, p, table8, theta, s, tab, mask, cut, st);
    } else if (p.nq == 64) {
        launch_excess<16>(ix, p, table8, theta, s, tab, mask, cut, st);
    } else {
        const int gy = batch_groups(p) * group / 8;
        int64_t gx = (8LL * ix.sm_count + gy - 1) / gy;
        if (gx > (ix.K + 8) / 8) gx = (ix.K + 8) / 8;
        launch(p.nq <= 32 ? batch_excess_exact_kernel<1> : p.nq <= 64 ? batch_excess_exact_kernel<2> : batch_excess_exact_kernel<4>,
               dim3((unsigned)gx, (unsigned)gy), BS_THREADS, 0, st, table, ix.K, p.nq, p.B, group, theta, us, s.scale, table8, tab,
               s.n_over, s.over, (uint8_t *)mask);
    }
    CHIMERA_CUDA(cudaGetLastError());
    auto scan = group == 8     ? launch_scan<1, 2, 1, 4>
                : group == 16  ? launch_scan<1, 4, 1, 4>
                : group == 32  ? launch_scan<2, 4, 1, 4>
                : group == 64  ? launch_scan<4, 4, 1, 8>
                : group == 128 ? launch_scan<8, 4, 2, 8>
                               : launch_scan<16, 4, 2, 8>;
    scan(ix, p, tab, ranks, L.words, s.scale, hi0, cut, st);
    CHIMERA_CUDA(cudaGetLastError());
    int64_t gx = (16LL * ix.sm_count + p.B - 1) / p.B;
    if (gx > 3 * p.nq) gx = 3 * p.nq;
    launch(!wide ? batch_over_kernel<0> : p.nq == 32 ? batch_over_kernel<8> : batch_over_kernel<16>, dim3((unsigned)gx, (unsigned)p.B),
           BS_THREADS, 0, st, table, table8, ix.K, p.nq, theta, us, s.scale, s.n_over, s.over, ix.ivf_off, ix.ivf_doc, ranks, L.words,
           p.maxc, hi0, cut);
    CHIMERA_CUDA(cudaGetLastError());
    gx = (4LL * ix.sm_count + p.B - 1) / p.B;
    if (gx > (p.maxc + 8191) / 8192) gx = (p.maxc + 8191) / 8192;
    launch(batch_hist_kernel, dim3((unsigned)gx, (unsigned)p.B), SEL_THREADS, 0, st, hi0, n_cand, p.maxc, s.scale, us,
           (int32_t *)(ws + L.flt_hist), cut);
    CHIMERA_CUDA(cudaGetLastError());
    count_launch(SLOT_CI, 4);
    return CHIMERA_OK;
}

}  // namespace chimera
