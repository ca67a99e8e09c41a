// Stage 3, first cut: an upper bound on CI from ONE number per document token, so that the row lookups of the later
// phases (g3_centroid_interaction.cu) run over a small part of the candidates only.
//
// For any thresholds theta_i,  max_t S[c_t, i] <= theta_i + sum_t (S[c_t, i] - theta_i)+ , so with
//     e(c) = sum_i (S[c, i] - theta_i)+                    (one number per centroid and query)
//     CI(d) = sum_i max_t S[c_t, i]  <=  sum_i theta_i + sum_t e(c_t) = hi0(d).
// theta_i is set so that about FILTER_LAMBDA of a document's tokens exceed it: lower thresholds count a column's second
// and third best tokens as well, higher ones replace the column's true maximum by theta.  Any choice is correct; with one
// token per column of a long document of independent tokens the bound keeps 7-13 % of the candidates when 1 % are wanted
// (65,536 and 262,144 centroids, candidates of 85-512 tokens), with half or one and a half times as many up to twice that.
//
// With documents that repeat their centroids, or hold several near the same query token, the bound counts each of them where
// CI counts one, and most candidates pass it; then the cut only costs (below, at filter_sample_kernel).
//
//   filter_theta_kernel    theta_i from a sample of the table's rows
//   filter_sample_kernel    q_len 32 / 64: whether the cut would drop enough, from sampled candidates; if not, the kernels
//                          down to the count return at once, all candidates are kept, and their 8-bit bounds decide
//   filter_excess_kernel   e(c) of every centroid, rounded up (16 bits, or 6-bit codes five to a word for large K), and a mask
//                          of those where it is not zero
//   filter_scan_kernel     hi0 of every candidate: the query's whole e table in shared memory, one lookup per token
//                          (batches whose candidates are a good part of the corpus: all queries at once, g3_batch_scan.cu)
//   filter_seed_kernel     the ~2 n_prune candidates with the largest hi0 (their order does not matter)
//   (their exact CI: g3_centroid_interaction.cu)
//   filter_count_kernel,   tau = the n_prune-th largest of those, a lower bound on the n_prune-th largest CI; keeps every
//   filter_write_kernel    candidate with hi0 >= tau, ascending, with its token range
//   (upper bounds of the kept ones from the 8-bit table, of few tokens first: g3_centroid_interaction.cu)
//   filter_contend_kernel  and of those the ones whose bound reaches tau
//   (exact CI of what is left, except for the seeds, and the exact selection: g3_centroid_interaction.cu)
// Every document of the exact top n_prune has an upper bound >= CI >= tau, so it is never dropped and the result is the
// same as without these cuts.
#include <limits.h>
#include <math.h>

#include "g3_filter.cuh"

namespace chimera {

constexpr double FILTER_LAMBDA = 1.0;     // wanted tokens of a document above theta, per query token
constexpr int FILTER_SAMPLE = 4096;       // table rows sampled per query for theta
constexpr int KEEP_SPLIT = 32;            // most blocks per query of the selection kernels
constexpr int CUT_KEPT_PERCENT = 58;        // of the sampled candidates: with more the call does without the cut
constexpr int64_t FILTER_SMEM = 208 * 1024;   // shared memory of the scan's block that its e table may take

// 6-bit codes of e in units of 2^16 (1/256): exact up to 20, then steps of about 7 % (the sums of a document's far
// tokens are 1-30, a token of a probed centroid adds about 180), a few large ones for centroids near several query
// tokens, and the largest possible value (127 * 257).
struct FilterLevels { uint16_t v[64]; };
constexpr FilterLevels filter_levels()
{
    FilterLevels l{};
    for (int j = 0; j <= 20; ++j) l.v[j] = (uint16_t)j;
    for (int j = 21; j < 60; ++j) l.v[j] = (uint16_t)(l.v[j - 1] + (l.v[j - 1] * 19 >> 8) + 1);
    l.v[60] = 1024; l.v[61] = 2048; l.v[62] = 8192; l.v[63] = 32640;
    return l;
}
__constant__ FilterLevels c_levels = filter_levels();

// How the e table of a query is kept: 16 = 16-bit values (K <= 106,496), 6 = 6-bit codes (K <= 266,240), 0 = not at all.
static int filter_codec(int64_t K)
{
    if (K * 2 <= FILTER_SMEM) return 16;
    if ((K + 4) / 5 * 4 <= FILTER_SMEM) return 6;
    return 0;
}

// When the cut runs.  The table has to fit one SM's shared memory; a token position has to fit 32 bits and a document's
// sum of e 31 bits; and there has to be enough to scan that the cut pays for its launches (14 against 8 kernels for q_len
// 32 / 64, whose other form scans 8-bit rows, 11 against 6 for the others, which look up exact rows), for its tables (per
// query and centroid) and for the exact rows of its seeds.  What is scanned is what the candidates hold, so their expected
// number counts and not the room for them; a document is a candidate when one of its distinct centroids is probed.
// In tokens, per query, fitted to calls with and without the cut (independent tokens, kept 1-60 %; within 4 % of the better
// form in 70 of 74 calls on 2,000 to 1.5 million documents, and the others lose at most a quarter):
//   q_len 32 / 64: 8 per centroid, 5 n_prune documents, 20 M a call.  Mid's documents, one query, 12 M tokens: 206 us with
//     the cut, 187 without; two: 248 / 266; eight: 537 / 720; 64 queries with one probe a token on 4 million documents and
//     262,144 centroids, 2.2 M tokens each: 2,451 / 2,300; with four probes, 8.7 M each: 32 queries 2,746 / 3,103, two 414 / 372.
//   others: 4 per centroid, 4 n_prune documents, 2 M a call.  21 tokens, 20,000 documents, 1.3 M tokens: 143 us with the cut, 133
//     without; 2.6 M: 153 / 181; 100 tokens on 200,000 documents, 12 M: 263 / 756.
double expected_candidates(const Index &ix, const Params &p)
{
    const double distinct = (double)ix.ivf_len / (double)ix.N, probed = (double)p.nq * p.P / (double)ix.K;
    const double cand = probed < 1.0 ? (double)ix.N * (1.0 - pow(1.0 - probed, distinct)) : (double)ix.N;
    return cand < (double)p.maxc ? cand : (double)p.maxc;
}
double expected_tokens(const Index &ix, const Params &p)
{
    return expected_candidates(ix, p) * ((double)ix.T / (double)ix.N);
}
// Share of the centroids above each threshold: FILTER_LAMBDA tokens of a document.  Its length is that of the documents that
// compete for the top: about halfway between the candidates' mean (somewhat above the corpus's: long documents are probed more
// often) and the longest, outliers aside.
static double filter_share(const Index &ix)
{
    const double mean = (double)ix.T / (double)ix.N, most = (double)ix.max_doclen;
    const double len = 0.5 * ((1.2 * mean < most ? 1.2 * mean : most) + (2.4 * mean < most ? 2.4 * mean : most));
    return FILTER_LAMBDA / len;
}
// Whether the bounds of what is kept start with the tokens near the query (ci_bound_kernel).  Measured as the time of the step, all
// rows at once / near tokens first (independent tokens unless said):
//   Tokens near, as the thresholds are set: with more than four tenths of them the other columns are too many for a bound that
//     decides.  64 queries, n_prune 2,048, by the share: 32 query tokens 0.30 301 / 283 us, 0.39 264 / 249, 0.44 255 / 267, 0.66 212 / 219; 64:
//     0.47 783 / 748, 0.59 669 / 682; 100: 0.31 2,130 / 1,850, 0.41 1,865 / 1,833, 0.53 1,535 / 1,646, 0.74 1,342 / 1,589.
//   Documents looked at: each is a chain of lookups whose length does not shrink with the rows, and there is a second kernel.
//     B n_prune from 65,536 on nothing of 32 tokens or more lost more than 10 % (topics, most of them kept), and most gained 5 to 35 %:
//     Mid, 64 queries, n_prune 1,024, 308 / 263; 64 tokens on 512-token documents, 64 queries, n_prune 1,024, 890 / 576; 100 tokens on
//     those, 64 queries, 2,048, 3,886 / 2,608.  Below, it goes by the documents: 32,768: 200 / 203, 165 / 150 (Mid, n_prune 256 and 512),
//     475 / 336 (64 tokens); 16,384: 101 / 118, 89 / 74, 322 / 294, and 302 / 458 with 60 tokens, 1,151 / 2,040 with 110.
//   Fewer than 32 query tokens: the bound of a document is a sum of few columns, and those that pass cost both kernels.  Mid, 64
//     queries, n_prune 2,048: 8 tokens 124 / 159, 16: 258 / 291, 21: 356 / 376, 28: 452 / 449; documents of four topics 461 / 595, 1,088 /
//     1,472, 1,174 / 1,601, 1,657 / 2,123.  (32 tokens: 504 / 435; topics that keep most of them do without the cut.)
// (6-bit codes from the exact table come five centroids to a warp: no words of a mask.)
bool filter_mask_used(const Index &ix, const Params &p, bool batch)
{
    return p.nq >= 32 && filter_share(ix) * p.nq < 0.4 && (int64_t)p.B * p.n_prune >= 65536 &&
           (batch || coarse_supported(p.nq) || filter_codec(ix.K) == 16);
}
bool filter_used(const Index &ix, const Params &p)
{
    if (filter_codec(ix.K) == 0 || ix.T >= 0x7fffff00LL || ix.max_doclen > 32000) return false;
    const bool wide = coarse_supported(p.nq);
    const double len = (double)ix.T / (double)ix.N;
    const double fixed = (wide ? 8.0 : 4.0) * (double)ix.K + (wide ? 5.0 : 4.0) * p.n_prune * len;
    return (double)p.B * (expected_tokens(ix, p) - fixed) >= (wide ? 2e7 : 2e6);
}
size_t filter_table_pitch(const Index &ix)
{
    const int codec = filter_codec(ix.K);
    const size_t bytes = codec == 16 ? (size_t)ix.K * 2 : codec == 6 ? (size_t)(ix.K + 4) / 5 * 4 : 0;
    return (bytes + 15) & ~(size_t)15;
}
int filter_hist_bins() { return FILTER_BINS; }
int filter_count_slots() { return KEEP_SPLIT; }
// Blocks per query of the selection kernels: slices of 4,096 candidates or more, and no more blocks than are resident at once
// (two of 1,024 threads per SM): every block of a query first finds tau, or the seeds' histogram bin, for itself, so a second
// wave costs as much as the first (256 queries in 3 x 256 blocks: 214 us for the keep steps, in 256: 183).
static int filter_split(const Index &ix, const Params &p)
{
    int64_t g = 2LL * ix.sm_count / p.B;
    if (g > (p.maxc + 4095) / 4096) g = (p.maxc + 4095) / 4096;
    return (int)(g > KEEP_SPLIT ? KEEP_SPLIT : g < 1 ? 1 : g);
}

// Queries that are sampled, candidates of each, and what the kernels behind it go by.
static int cut_queries(const Params &p) { return p.B < CUT_QUERIES ? p.B : CUT_QUERIES; }
static int cut_samples(const Params &p) { return CUT_SAMPLES / 32 / cut_queries(p) * 32; }
FirstCut first_cut(const Params &p, const Layout &L, char *ws)
{
    FirstCut c;
    c.kept = coarse_supported(p.nq) ? (const int32_t *)(ws + L.flt_vote) : nullptr;
    c.most = cut_queries(p) * cut_samples(p) * CUT_KEPT_PERCENT / 100;
    return c;
}

// Blocks per query and column group of the theta kernel, and the bytes they share.
static int filter_parts(const Index &ix, const Params &p) { return 4 * p.B <= ix.sm_count ? 8 : 1; }
size_t filter_parts_bytes(const Index &ix, const Params &p)
{
    return filter_parts(ix, p) > 1 ? sizeof(int32_t) * (size_t)p.B * ((p.nq + 31) / 32) * (256 * 32 + 1) : 0;
}

// ------------------------------------------------------------------------------------------------ thresholds ------
// grid (ceil(nq / 32), B, parts), lane = query token.  theta[b][i] = the smallest t (in units of 2^16) such that at most
// `rank` of the m sampled rows (every step-th one) have S >= t 2^16.  With few queries the sample is split over several
// blocks that add their histograms up in `parts_hist` ([B][groups][256 * 32], cleared before); the last one to
// finish (`done`, likewise) reads the sum.  Also clears what the scan and the seed selection add to, and the sample's words (vote,
// may be NULL).  Row: uint8_t, of the 8-bit table, which holds all that is read here in a quarter of the bytes, or int32_t (a choice made
// at each load instead of by the type cost the latter a third: 120 tokens, 31 queries 59 -> 72 us).
template <class Row>
__global__ void __launch_bounds__(SEL_THREADS)
filter_theta_kernel(const Row *__restrict__ table, int64_t K, int nq, int m, int step, int rank,
                    int32_t *__restrict__ theta, int32_t *__restrict__ hist_out, int32_t *__restrict__ n_seed,
                    int32_t *__restrict__ parts_hist, int32_t *__restrict__ done, int32_t *__restrict__ vote)
{
    pdl_entry();
    __shared__ int hist[256 * 32];
    __shared__ int s_last;
    if (vote && blockIdx.x == 0 && blockIdx.y == 0 && blockIdx.z == 0 && threadIdx.x < 64) vote[threadIdx.x] = 0;
    const int b = blockIdx.y, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int col = blockIdx.x * 32 + lane;
    for (int i = threadIdx.x; i < 256 * 32; i += SEL_THREADS) hist[i] = 0;
    if (blockIdx.x == 0 && blockIdx.z == 0) {
        for (int i = threadIdx.x; i < FILTER_BINS; i += SEL_THREADS) hist_out[(int64_t)b * FILTER_BINS + i] = 0;
        if (threadIdx.x == 0) n_seed[b] = 0;
    }
    __syncthreads();
    const Row *tb = table + (int64_t)b * K * nq + col;
    const int64_t row = (int64_t)step * nq;
    for (int r0 = blockIdx.z * 32 + warp; r0 < m; r0 += gridDim.z * 32 * 16) {
        int k[16];
#pragma unroll
        for (int u = 0; u < 16; ++u) {
            const int r = r0 + gridDim.z * 32 * u;
            k[u] = r >= m || col >= nq ? 0 : sizeof(Row) == 1 ? (int)tb[r * row] : (int)tb[r * row] >> 16;
        }
#pragma unroll
        for (int u = 0; u < 16; ++u)
            if (k[u] > 0) atomicAdd(&hist[(k[u] > 255 ? 255 : k[u]) * 32 + lane], 1);
    }
    __syncthreads();
    if (gridDim.z > 1) {
        int32_t *ph = parts_hist + ((int64_t)b * gridDim.x + blockIdx.x) * 256 * 32;
        for (int i = threadIdx.x; i < 256 * 32; i += SEL_THREADS)
            if (hist[i]) atomicAdd(&ph[i], hist[i]);
        __threadfence();
        __syncthreads();
        if (threadIdx.x == 0) s_last = atomicAdd(&done[(int64_t)b * gridDim.x + blockIdx.x], 1) == (int)gridDim.z - 1;
        __syncthreads();
        if (!s_last) return;
        __threadfence();
        for (int i = threadIdx.x; i < 256 * 32; i += SEL_THREADS) hist[i] = __ldcg(&ph[i]);
        __syncthreads();
    }
    // warp w finds column w's threshold: lane l holds buckets 255 - 8 l ... 248 - 8 l, descending
    int h[8], mine = 0;
#pragma unroll
    for (int e = 0; e < 8; ++e) { h[e] = hist[(255 - 8 * lane - e) * 32 + warp]; mine += h[e]; }
    int incl = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += t;
    }
    int above = incl - mine, best = 256;                     // the lowest t whose count is within the rank
#pragma unroll
    for (int e = 0; e < 8; ++e) {
        above += h[e];
        if (above <= rank) best = 255 - 8 * lane - e;
    }
    best = __reduce_min_sync(0xffffffffu, best);
    if (best < 1) best = 1;
    if (lane == 0 && blockIdx.x * 32 + warp < nq) theta[(int64_t)b * nq + blockIdx.x * 32 + warp] = best;
}

// ------------------------------------------------------------------------------------------------ sample ----------
// Does the cut pay?  CUT_SAMPLES candidates, spread over up to CUT_QUERIES queries of the call: CI from the 8-bit rows
// and the bound hi0, then the share of them whose bound reaches the sample's own n_prune-th of n_cand.  A query with so few
// candidates that all are kept counts as kept.  Queries of a batch search the same documents, so one answer per call is
// enough, and results do not depend on it.
// Where the line lies (batches of Mid's sizes unless said; the share that passes, with the cut / without it): documents that
// draw a quarter as many centroids as they have tokens (100 %): 8.09 / 6.36 ms; of neighbouring centroids of four topics (63 %,
// by the sample 57 %): 9.76 / 9.21, 16 queries (66 %, by the sample 60 %): 1,034 / 873 us; 512 tokens of such (35 %, sample 27 %):
// 25.7 / 28.7 ms; independent centroids, 16 queries, n_prune 16,384 (55 %, sample 56 %): 2.96 / 3.04 ms.  As the sample decides: 6.46
// ms, 9.73 ms, 915 us, 25.8 ms and 2.96 ms.  It costs 15 us where the cut stays (16 queries: 809 -> 825 us; 64 of 64 tokens on
// 512-token documents 30 of 12,740), most of it latency: candidate, range, ids, rows, then the last block's histogram (4 us).  Half as many
// samples, eight rows in flight per lane, or four warps per document are no faster.
// grid (blocks, queries), a document per warp, sixteen columns per lane, 64 tokens in flight.
template <int NQ>
__global__ void __launch_bounds__(SEL_THREADS)
filter_sample_kernel(const uint8_t *__restrict__ table8, int64_t K, const int32_t *__restrict__ theta, int B,
                    const int32_t *__restrict__ cand, const int32_t *__restrict__ n_cand, int64_t maxc,
                    const int64_t *__restrict__ doc_off, const int32_t *__restrict__ cids, int n_prune, bool coded,
                    const int2 *__restrict__ scale, int2 *__restrict__ smp, int32_t *__restrict__ vote)
{
    pdl_entry();
    constexpr int LPR = NQ / 16;                             // lanes per row, 16 columns each
    constexpr int TPL = 32 / LPR;                            // rows per load of the warp
    constexpr int BINS = 2048;                               // of 8 units: CI <= 64 (255 + 1/2)
    __shared__ int hist[BINS];
    __shared__ int warp_part[32];
    __shared__ int s_last, s_bin;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, sub = lane % LPR, grp = lane / LPR;
    const int b = (int)((int64_t)blockIdx.y * B / gridDim.y), m = (int)gridDim.x * 32;
    const int n = n_cand[b];
    int32_t *ticket = vote + 1 + blockIdx.y;
    int2 *mine = smp + (int64_t)blockIdx.y * m;
    const bool few = n <= 2 * n_prune + 32;
    if (!few) {
        const int s = blockIdx.x * 32 + warp;
        const int2 r = doc_range(doc_off, cand[(int64_t)b * maxc + (int64_t)s * n / m]);
        const uint4 *tb = reinterpret_cast<const uint4 *>(table8 + (int64_t)b * K * NQ) + sub;
        uint2 tm1[4];                                        // thresholds minus one, as in filter_row_excess
        int sum_tm1 = 0;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int4 t = __ldg(reinterpret_cast<const int4 *>(theta + (int64_t)b * NQ + 16 * sub) + k);
            tm1[k] = make_uint2((uint32_t)(t.x - 1) | (uint32_t)(t.z - 1) << 16, (uint32_t)(t.y - 1) | (uint32_t)(t.w - 1) << 16);
            sum_tm1 += t.x + t.y + t.z + t.w - 4;
        }
        uint32_t best[4] = {0u, 0u, 0u, 0u};
        int over = 0, above = 0;                             // sum of e and tokens that have one
        int32_t cid[2];                                      // 64 tokens at a time
#pragma unroll
        for (int h = 0; h < 2; ++h) cid[h] = 32 * h + lane < r.y ? cids[r.x + 32 * h + lane] : 0;
        for (int t0 = 0; t0 < r.y; t0 += 64) {
            uint4 v[2 * LPR];
#pragma unroll
            for (int u = 0; u < 2 * LPR; ++u) {
                const int64_t c = DBG_CID(__shfl_sync(0xffffffffu, cid[u / LPR], u % LPR * TPL + grp));
                v[u] = t0 + u * TPL + grp < r.y ? __ldg(tb + c * LPR) : make_uint4(0u, 0u, 0u, 0u);
            }
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int t = t0 + 64 + 32 * h + lane;
                cid[h] = t < r.y ? cids[r.x + t] : 0;
            }
#pragma unroll
            for (int u = 0; u < 2 * LPR; ++u) {
                const uint32_t w[4] = {v[u].x, v[u].y, v[u].z, v[u].w};
                uint32_t acc = 0;                            // 16-bit fields of at most 8 * 255
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    best[k] = __vmaxu4(best[k], w[k]);
                    acc += __vmaxu2(w[k] & 0x00ff00ffu, tm1[k].x) + __vmaxu2((w[k] >> 8) & 0x00ff00ffu, tm1[k].y);
                }
                const int e = (int)(acc & 0xffffu) + (int)(acc >> 16) - sum_tm1;
                over += e;
                above += e > 0 ? 1 : 0;
            }
        }
        int ci = 0;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
#pragma unroll
            for (int o = LPR; o < 32; o <<= 1) best[k] = __vmaxu4(best[k], __shfl_xor_sync(0xffffffffu, best[k], o));
            ci += (int)__vsadu4(best[k], 0u);
        }
        ci = __reduce_add_sync(0xffffffffu, lane < LPR ? ci : 0) + NQ / 2;
        over = __reduce_add_sync(0xffffffffu, over);
        const int base = __reduce_add_sync(0xffffffffu, lane < LPR ? sum_tm1 : 0) + NQ;
        // codes round up: the scan by query's by half a step of 7 % on average, the batch's by half a step of the query's
        if (scale) over += __reduce_add_sync(0xffffffffu, above) * (scale[b].y - 1) / 2;
        else if (coded) over += over / 28;
        if (lane == 0) mine[s] = make_int2(ci, base + over);
    }
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) s_last = atomicAdd(ticket, 1) == (int)gridDim.x - 1;
    __syncthreads();
    if (!s_last) return;                                     // the query's last block goes on
    __threadfence();
    int kept = m;
    if (!few) {
        for (int i = threadIdx.x; i < BINS; i += SEL_THREADS) hist[i] = 0;
        __syncthreads();
        for (int i = threadIdx.x; i < m; i += SEL_THREADS) atomicAdd(&hist[min(__ldcg(&mine[i].x) >> 3, BINS - 1)], 1);
        __syncthreads();
        int want = (int)(((int64_t)m * n_prune + n / 2) / n);
        if (want < 1) want = 1;
        const int hi_bin = BINS - 1 - 2 * (int)threadIdx.x;
        const int h_hi = hist[hi_bin], h_lo = hist[hi_bin - 1];
        int total;
        const int before = sel_block_scan(h_hi + h_lo, &total, warp_part);
        if (before < want && want <= before + h_hi + h_lo) s_bin = want <= before + h_hi ? hi_bin : hi_bin - 1;
        __syncthreads();
        int pass = 0;
        for (int i = threadIdx.x; i < m; i += SEL_THREADS) pass += __ldcg(&mine[i].y) >= s_bin << 3 ? 1 : 0;
        sel_block_scan(pass, &kept, warp_part);
    }
    if (threadIdx.x == 0) atomicAdd(&vote[0], kept);
}

// ------------------------------------------------------------------------------------------------ excess table ----
// Smallest code whose level is >= e.
__device__ __forceinline__ int filter_encode(const uint8_t *enc, int e)
{
    return e < 512 ? enc[e] : e <= 1024 ? 60 : e <= 2048 ? 61 : e <= 8192 ? 62 : 63;
}
__device__ __forceinline__ void filter_fill_encoder(uint8_t *enc)
{
    for (int e = threadIdx.x; e < 512; e += blockDim.x) {
        int j = 0;
        while (c_levels.v[j] < e) ++j;
        enc[e] = (uint8_t)j;
    }
    __syncthreads();
}

// grid (blocks, B).  One thread per centroid (16-bit values) or per five centroids (6-bit codes): a stream of the 8-bit
// table (Mid, batch 256: 537 MB).
template <int WORDS, int CODEC>
__global__ void __launch_bounds__(256)
filter_excess_kernel(const uint8_t *__restrict__ table8, int64_t K, const int32_t *__restrict__ theta,
                     uint8_t *__restrict__ out, size_t pitch, uint32_t *__restrict__ mask, FirstCut cut)
{
    pdl_entry();
    __shared__ uint2 tm1[WORDS];
    __shared__ uint32_t s_bits[2][CODEC == 6 ? 40 : 1];      // of 256 words of five codes
    __shared__ int s_sum;
    __shared__ uint8_t enc[512];
    const int b = blockIdx.y;
    const int32_t *th = theta + (int64_t)b * 4 * WORDS;
    if (!cut.on()) return;
    if (threadIdx.x < WORDS) {
        const int32_t *t = th + 4 * threadIdx.x;
        tm1[threadIdx.x] = make_uint2((uint32_t)(t[0] - 1) | (uint32_t)(t[2] - 1) << 16,
                                      (uint32_t)(t[1] - 1) | (uint32_t)(t[3] - 1) << 16);
    }
    if (threadIdx.x == 0) {
        int s = 0;
        for (int i = 0; i < 4 * WORDS; ++i) s += th[i] - 1;
        s_sum = s;
    }
    if (CODEC == 6) filter_fill_encoder(enc);
    __syncthreads();
    const uint4 *tb = reinterpret_cast<const uint4 *>(table8 + (int64_t)b * K * 4 * WORDS);
    uint8_t *ob = out + (size_t)b * pitch;
    const int sum = s_sum;
    uint32_t *mb = mask + (int64_t)b * ((K + 31) / 32);
    if (CODEC == 16) {
        for (int64_t c0 = (int64_t)blockIdx.x * 256; c0 < K; c0 += (int64_t)gridDim.x * 256) {
            const int64_t c = c0 + threadIdx.x;
            const int e = c < K ? filter_row_excess<WORDS>(tb + c * (WORDS / 4), tm1, sum) : 0;
            if (c < K) reinterpret_cast<uint16_t *>(ob)[c] = (uint16_t)e;
            const uint32_t bits = __ballot_sync(0xffffffffu, e > 0);
            if ((threadIdx.x & 31) == 0 && c < K) mb[c >> 5] = bits;
        }
    } else {
        const int64_t words = (K + 4) / 5;
        if (threadIdx.x < 40) s_bits[0][threadIdx.x] = 0u;
        __syncthreads();
        int buf = 0;
        for (int64_t w0 = (int64_t)blockIdx.x * 256; w0 < words; w0 += (int64_t)gridDim.x * 256, buf ^= 1) {
            const int64_t w = w0 + threadIdx.x;
            if (threadIdx.x < 40) s_bits[buf ^ 1][threadIdx.x] = 0u;
            if (w < words) {
                uint32_t packed = 0, bits = 0;
#pragma unroll
                for (int r = 0; r < 5; ++r) {
                    const int64_t c = w * 5 + r < K ? w * 5 + r : K - 1;
                    const int e = filter_row_excess<WORDS>(tb + c * (WORDS / 4), tm1, sum);
                    packed |= (uint32_t)filter_encode(enc, e) << (6 * r + (r > 2));
                    bits |= (uint32_t)(e > 0) << r;
                }
                reinterpret_cast<uint32_t *>(ob)[w] = packed;
                const int at = 5 * threadIdx.x;
                atomicOr(&s_bits[buf][at >> 5], bits << (at & 31));
                if ((at & 31) > 27) atomicOr(&s_bits[buf][(at >> 5) + 1], bits >> (32 - (at & 31)));
            }
            __syncthreads();                             // (the next round clears and fills the other half)
            const int64_t mw = w0 * 5 / 32 + threadIdx.x;
            if (threadIdx.x < 40 && mw < (K + 31) / 32) mb[mw] = s_bits[buf][threadIdx.x];
        }
    }
}

// The same from the exact table, for any q_len: one warp per row, values rounded up to units of 2^us (a score that reaches theta
// counts, so that zero means a centroid with none).  The 8-bit rows that
// the second bound looks up are made on the way (table8: [B][K][pitch8], a lane's columns side by side, zeros for those
// past nq: the bound is a sum over columns, whatever their order).
template <int CODEC, int NQW>      // NQW = pitch8 / 32
__global__ void __launch_bounds__(256)
filter_excess_exact_kernel(const int32_t *__restrict__ table, int64_t K, int nq, const int32_t *__restrict__ theta, int us,
                           uint8_t *__restrict__ table8, uint8_t *__restrict__ out, size_t pitch, uint8_t *__restrict__ mask)
{
    pdl_entry();
    __shared__ uint8_t enc[512];
    if (CODEC == 6) filter_fill_encoder(enc);
    const int b = blockIdx.y, lane = threadIdx.x & 31;
    constexpr int pitch8 = 32 * NQW;
    uint8_t *t8 = table8 + (int64_t)b * K * pitch8;
    int th[NQW];
#pragma unroll
    for (int w = 0; w < NQW; ++w) th[w] = lane + 32 * w < nq ? (theta[(int64_t)b * nq + lane + 32 * w] << 16) - 1 : 0;
    const int32_t *tb = table + (int64_t)b * K * nq;
    uint8_t *ob = out + (size_t)b * pitch;
    constexpr int PER = CODEC == 16 ? 8 : 5;                          // rows per warp and iteration
    const int64_t groups = (K + PER - 1) / PER;
    for (int64_t g = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5); g < groups; g += (int64_t)gridDim.x * 8) {
        int e[PER];
        uint32_t coarse[PER];
#pragma unroll
        for (int r = 0; r < PER; ++r) { e[r] = 0; coarse[r] = 0u; }
#pragma unroll
        for (int w = 0; w < NQW; ++w) {
            int v[PER];
#pragma unroll
            for (int r = 0; r < PER; ++r)
                v[r] = (lane + 32 * w < nq && g * PER + r < K) ? __ldg(tb + (g * PER + r) * nq + lane + 32 * w) : 0;
#pragma unroll
            for (int r = 0; r < PER; ++r) {
                coarse[r] |= (uint32_t)__vimin_s32_relu(v[r] >> 16, 255) << (8 * w);
                e[r] += max(v[r] - th[w], 0);     // (a column past the end has neither a value nor a threshold)
            }
        }
#pragma unroll
        for (int r = 0; r < PER; ++r) {
            if (g * PER + r >= K) break;
            uint8_t *row = t8 + (g * PER + r) * pitch8;
            if constexpr (NQW == 1) row[lane] = (uint8_t)coarse[r];
            else if constexpr (NQW == 2) reinterpret_cast<uint16_t *>(row)[lane] = (uint16_t)coarse[r];
            else reinterpret_cast<uint32_t *>(row)[lane] = coarse[r];
        }
        uint32_t packed = 0, near = 0;
        int val = 0;
#pragma unroll
        for (int r = 0; r < PER; ++r) {
            // the sum of 127 columns stays below 2^31; + the rounding, so add in unsigned
            const uint32_t s = ((uint32_t)__reduce_add_sync(0xffffffffu, e[r]) + ((1u << us) - 1)) >> us;
            near |= (uint32_t)(s > 0) << r;
            if (CODEC == 16) { if (lane == r) val = (int)s; }
            else packed |= (uint32_t)filter_encode(enc, (int)s) << (6 * r + (r > 2));
        }
        if (CODEC == 16) {
            if (lane < PER && g * PER + lane < K) reinterpret_cast<uint16_t *>(ob)[g * PER + lane] = (uint16_t)val;
            if (NQW > 1 && lane == 0) mask[(int64_t)b * ((K + 31) / 32) * 4 + g] = (uint8_t)near;    // (filter_mask_used)
        } else if (lane == 0) {
            reinterpret_cast<uint32_t *>(ob)[g] = packed;
        }
    }
}

// ------------------------------------------------------------------------------------------------ scan ------------
// grid (blocks per query, B), one block of 1,024 threads per SM, the query's e table in shared memory.  Eight lanes take
// a document: each loads four consecutive centroid ids with one 16-byte load (a group reads a 128-byte line), looks
// the four up in shared memory (32 random banks: about 3.5 wavefronts per 32 tokens, against one L1 line per token for
// the row lookups of the later phases) and adds.  A warp holds four documents and has the loads of its next 64 tokens
// per document -- of the same documents or of the next four -- in flight while the present ones are looked up.
// The instruction pipe is the limit, so lanes must not idle: the block takes its candidates in windows of 1,024, one
// thread per candidate finds the token range (loads issued a window ahead), and a counting sort by number of 32-token
// chunks gives every warp four documents of about the same length.
//   hi0   [B][maxc]         sum_i theta_i + sum_t e(c_t) in units of 2^us
//   hist  [B][FILTER_BINS]  of sum_t e(c_t) in units of 2^17
constexpr int SCAN_THREADS_F = 1024;
constexpr int SCAN_SORT_BINS = 64;

template <int CODEC>
__global__ void __launch_bounds__(SCAN_THREADS_F, 1)
filter_scan_kernel(const uint8_t *__restrict__ tab, size_t pitch, const int32_t *__restrict__ theta, int nq, int us,
                   const int32_t *__restrict__ cand, const int64_t *__restrict__ doc_off,
                   const int32_t *__restrict__ n_cand, int64_t maxc, const int32_t *__restrict__ cids, int64_t T,
                   int32_t *__restrict__ hi0, int32_t *__restrict__ hist, FirstCut cut)
{
    pdl_entry();
    extern __shared__ uint4 s_tab[];
    __shared__ uint16_t s_level[64];                     // two to a bank: no conflicts
    __shared__ int s_hist[FILTER_BINS];
    __shared__ int s_sort[SCAN_SORT_BINS];
    __shared__ uint2 s_rng[SCAN_THREADS_F];
    __shared__ uint16_t s_idx[SCAN_THREADS_F];
    __shared__ int s_theta;
    const int b = blockIdx.y, tid = threadIdx.x;
    const bool on = cut.on();
    const int n = n_cand[b];
    const int per = (n + (int)gridDim.x - 1) / (int)gridDim.x;
    const int j0 = blockIdx.x * per, j1 = j0 + per < n ? j0 + per : n;
    if (!on || j0 >= n) return;
    const int lane = tid & 31, warp = tid >> 5, grp = lane >> 3, sub = lane & 7;
    const int32_t *cb = cand + (int64_t)b * maxc;
    int32_t *out = hi0 + (int64_t)b * maxc;

    // token range of this thread's candidate of a window; an empty one past the end
    auto range_of = [&](int32_t d) {
        if (d < 0) return make_int2(0, 0);
        d = DBG_DOC(d);
        const int64_t t0 = __ldg(doc_off + d);
        return make_int2((int)t0, (int)(__ldg(doc_off + d + 1) - t0));
    };
    auto cand_of = [&](int base) { return base + tid < j1 ? __ldg(cb + base + tid) : -1; };
    int2 nx_rng = range_of(cand_of(j0));
    int32_t nx_cand = cand_of(j0 + SCAN_THREADS_F);

    const uint4 *src = reinterpret_cast<const uint4 *>(tab + (size_t)b * pitch);
#pragma unroll 4
    for (int i = tid; i < (int)(pitch / 16); i += SCAN_THREADS_F) s_tab[i] = __ldg(src + i);
    for (int i = tid; i < FILTER_BINS; i += SCAN_THREADS_F) s_hist[i] = 0;
    if (tid < 64) { s_level[tid] = c_levels.v[tid]; s_sort[tid] = 0; }
    if (tid < 32) {
        int s = 0;
        for (int i = tid; i < nq; i += 32) s += theta[(int64_t)b * nq + i];
        s = __reduce_add_sync(0xffffffffu, s);
        if (tid == 0) s_theta = s << (16 - us);
    }
    __syncthreads();
    const uint16_t *tab16 = reinterpret_cast<const uint16_t *>(s_tab);
    const uint32_t *tab6 = reinterpret_cast<const uint32_t *>(s_tab);

    // Positions count from the 16-byte boundary at or below cids.  Whole 16-byte groups inside the array are [edge_lo, edge_hi):
    // only the corpus's first and last documents can reach beyond, and the thread that owns one adds those tokens itself.
    const uint32_t mis = (uint32_t)(((uintptr_t)cids >> 2) & 3);
    const int4 *c4 = reinterpret_cast<const int4 *>(cids - mis);
    const uint32_t edge_lo = mis ? 4u : 0u, edge_hi = (mis + (uint32_t)T) & ~3u;
    auto load4 = [&](uint32_t q, uint32_t hi) { return q < hi ? __ldg(c4 + (q >> 2)) : make_int4(0, 0, 0, 0); };
    auto value = [&](int32_t c) -> int {
        c = DBG_CID(c);
        if (CODEC == 16) return tab16[c];
        // c / 5 in the high word, (c % 5) / 5 in the low one: its top five bits are the bit positions 0, 6, 12, 19, 25
        const unsigned long long pr = (unsigned long long)(uint32_t)c * 858993460u;
        return (int)s_level[(tab6[pr >> 32] >> ((uint32_t)pr >> 27)) & 63];
    };
    // the values of positions lead ... rem - 1 of a group of four
    auto add4 = [&](int acc, const int4 &v, int rem, int lead) {
        const int x = value(v.x), y = value(v.y), z = value(v.z), w = value(v.w);
        acc += rem > 0 && lead <= 0 ? x : 0;
        acc += rem > 1 && lead <= 1 ? y : 0;
        acc += rem > 2 && lead <= 2 ? z : 0;
        acc += rem > 3 ? w : 0;
        return acc;
    };

    for (int base = j0; base < j1; base += SCAN_THREADS_F) {
        const int cnt = j1 - base < SCAN_THREADS_F ? j1 - base : SCAN_THREADS_F;
        // counting sort by chunk count, long documents first
        const int2 r = nx_rng;
        nx_rng = range_of(nx_cand);
        nx_cand = cand_of(base + 2 * SCAN_THREADS_F);
        uint32_t lo = mis + (uint32_t)r.x, hi = lo + (uint32_t)r.y;
        int extra = 0;
        for (; lo < edge_lo && lo < hi; ++lo) extra += value(cids[lo - mis]);
        for (; hi > edge_hi && hi > lo; --hi) extra += value(cids[hi - 1 - mis]);
        if (hi <= lo) lo = hi = 0;
        int key = (int)((hi - (lo & ~3u) + 31) >> 5);
        key = SCAN_SORT_BINS - 1 - (key < SCAN_SORT_BINS ? key : SCAN_SORT_BINS - 1);
        int place = 0;
        if (tid < cnt) place = atomicAdd(&s_sort[key], 1);
        __syncthreads();
        if (warp == 0) {
            const int a = s_sort[2 * lane], c = s_sort[2 * lane + 1];
            int incl = a + c;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int t = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += t;
            }
            s_sort[2 * lane] = incl - a - c;
            s_sort[2 * lane + 1] = incl - c;
        }
        __syncthreads();
        if (tid < cnt) {
            place += s_sort[key];
            s_rng[place] = make_uint2(lo, hi);
            s_idx[place] = (uint16_t)tid;
        }
        __syncthreads();
        if (tid < SCAN_SORT_BINS) s_sort[tid] = 0;

        int k = warp * 4 + grp;
        uint2 cur = k < cnt ? s_rng[k] : make_uint2(0, 0);
        uint32_t q = (cur.x & ~3u) + 4 * sub;
        int4 a0 = load4(q, cur.y), a1 = load4(q + 32, cur.y);
        for (int kw = warp * 4; kw < cnt; kw += SCAN_THREADS_F / 8) {
            const int kn = k + SCAN_THREADS_F / 8;
            const uint2 nxt = kn < cnt ? s_rng[kn] : make_uint2(0, 0);
            const uint32_t qn = (nxt.x & ~3u) + 4 * sub;
            // steps of 64 tokens, as many as the longest of the four documents needs
            const int most = __reduce_max_sync(0xffffffffu, (int)(cur.y - (q - 4 * sub)));
            int acc = 0, rem = (int)(cur.y - q);
            int lead = sub == 0 ? (int)(cur.x & 3u) : 0;     // ids of the document before, in front of the first token
            for (int c = 0; c < most; c += 64) {
                int4 n0, n1;
                const bool last = c + 64 >= most;
                const uint32_t ql = last ? qn : q + 64, hl = last ? nxt.y : cur.y;
                n0 = load4(ql, hl);
                n1 = load4(ql + 32, hl);
                acc = add4(acc, a0, rem, lead);
                if (c + 32 < most) acc = add4(acc, a1, rem - 32, 0);
                lead = 0;
                rem -= 64;
                a0 = n0;
                a1 = n1;
                q = ql;
            }
            acc += __shfl_xor_sync(0xffffffffu, acc, 1);
            acc += __shfl_xor_sync(0xffffffffu, acc, 2);
            acc += __shfl_xor_sync(0xffffffffu, acc, 4);
            if (sub == 0 && k < cnt) {
                const int bin = acc >> (17 - us);
                atomicAdd(&s_hist[bin < FILTER_BINS ? bin : FILTER_BINS - 1], 1);
                out[base + s_idx[k]] = s_theta + acc;
            }
            k = kn;
            cur = nxt;
        }
        __syncthreads();
        if (extra > 0) out[base + tid] += extra;             // (the histogram keeps the smaller value: it only picks seeds)
    }
    int32_t *hb = hist + (int64_t)b * FILTER_BINS;
    for (int i = tid; i < FILTER_BINS; i += SCAN_THREADS_F)
        if (s_hist[i]) atomicAdd(&hb[i], s_hist[i]);
}

// ------------------------------------------------------------------------------------------------ seeds -----------
// A Q.24 threshold in units of 2^us, rounded up (hi0 is a whole number of them).
__device__ __forceinline__ int32_t units_up(int32_t tau, int us) { return (int32_t)(((long long)tau + (1 << us) - 1) >> us); }

// grid (split, B): candidates with the largest hi0, `want` of them and the rest of the last histogram bin, with their token
// ranges, in no particular order; seed_thr[b] = the hi0 they start at, seed_slot[candidate] = where each one went.  n_seed
// (cleared before) stays 0 when a query has so few candidates that all are kept.  A warp collects the places of the seeds that it
// meets, one in fifty, and looks up the documents of 32 at a time: one by one, each a chain of two reads, they took 129 us of Mid's
// batch of 256, now 57.
__global__ void __launch_bounds__(SEL_THREADS)
filter_seed_kernel(const int32_t *__restrict__ cand, const int32_t *__restrict__ n_cand, const int64_t *__restrict__ doc_off,
                   const int32_t *__restrict__ hi0, int64_t maxc, const int32_t *__restrict__ theta, int nq, int us,
                   const int32_t *__restrict__ hist, int want, int32_t *__restrict__ seed,
                   int2 *__restrict__ seed_rng, int32_t *__restrict__ n_seed, int32_t *__restrict__ seed_thr,
                   int32_t *__restrict__ seed_slot, FirstCut cut)
{
    pdl_entry();
    __shared__ int warp_part[32];
    __shared__ int s_bin, s_theta;
    __shared__ int32_t s_list[32][31 + 256];
    const bool on = cut.on();
    const int b = blockIdx.y, n = n_cand[b];
    if (!on) return;                                     // (no seeds: n_seed is 0)
    if (n <= want) {
        if (blockIdx.x == 0 && threadIdx.x == 0) seed_thr[b] = INT_MAX;
        return;
    }
    const int32_t *hb = hist + (int64_t)b * FILTER_BINS;
    constexpr int PER = FILTER_BINS / SEL_THREADS;
    const int first_bin = FILTER_BINS - 1 - PER * (int)threadIdx.x;
    int h[PER], mine = 0;
#pragma unroll
    for (int e = 0; e < PER; ++e) { h[e] = hb[first_bin - e]; mine += h[e]; }
    int total;
    int before = sel_block_scan(mine, &total, warp_part);
    if (before < want && want <= before + mine) {
#pragma unroll
        for (int e = 0; e < PER; ++e) {
            if (before < want && want <= before + h[e]) s_bin = first_bin - e;
            before += h[e];
        }
    }
    if (threadIdx.x < 32) {
        int s = 0;
        for (int i = threadIdx.x; i < nq; i += 32) s += theta[(int64_t)b * nq + i];
        s = __reduce_add_sync(0xffffffffu, s);
        if (threadIdx.x == 0) s_theta = s;
    }
    __syncthreads();
    const int32_t thr = (s_theta << (16 - us)) + (s_bin << (17 - us));
    if (blockIdx.x == 0 && threadIdx.x == 0) seed_thr[b] = thr;
    const int32_t *ub = hi0 + (int64_t)b * maxc;
    const int32_t *cb = cand + (int64_t)b * maxc;
    const int per = (n + (int)gridDim.x - 1) / (int)gridDim.x;
    const int j0 = blockIdx.x * per, j1 = j0 + per < n ? j0 + per : n;
    const int lane = threadIdx.x & 31;
    int32_t *list = s_list[threadIdx.x >> 5];
    int have = 0;
    auto flush = [&](int from, int many) {                   // list[from ... from + many), many <= 32
        int at = 0;
        if (lane == 0) at = atomicAdd(&n_seed[b], many);
        at = __shfl_sync(0xffffffffu, at, 0);
        if (lane < many) {
            const int j = list[from + lane];
            const int32_t d = cb[j];
            const int64_t o = (int64_t)b * maxc + at + lane;
            seed[o] = d;
            seed_slot[(int64_t)b * maxc + j] = at + lane;
            seed_rng[o] = doc_range(doc_off, d);
        }
    };
    for (int base = j0 + (threadIdx.x & ~31); base < j1; base += 8 * SEL_THREADS) {
        int32_t v[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const int j = base + u * SEL_THREADS + lane;
            v[u] = j < j1 ? ub[j] : INT_MIN;
        }
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const unsigned mask = __ballot_sync(0xffffffffu, v[u] >= thr);
            if (v[u] >= thr) list[have + __popc(mask & ((1u << lane) - 1))] = base + u * SEL_THREADS + lane;
            have += __popc(mask);
        }
        __syncwarp();
        if (have >= 32) {
            int from = 0;
            for (; have - from >= 32; from += 32) flush(from, 32);
            have -= from;
            const int32_t rest = lane < have ? list[from + lane] : 0;
            __syncwarp();
            if (lane < have) list[lane] = rest;              // (the places behind are written next, by other lanes)
        }
    }
    __syncwarp();
    if (have > 0) flush(0, have);
}

// ------------------------------------------------------------------------------------------------ keep ------------
// Ordered compaction of a slice [j0, j1) by a whole block: every element with v >= thr, in order.  A warp takes 256
// consecutive elements per round (eight coalesced loads), one block scan per 8,192.  The places of those that are kept go through
// shared memory (KEEP_ROUND entries), so that emit(j, position) runs on neighbouring positions in neighbouring threads: its chains
// of reads (document, offsets) are then as many as the threads and not one after the other (Mid, batch 256, 12 % kept: 112 -> 71 us).
constexpr int KEEP_ROUND = 8 * SEL_THREADS;
template <class Emit>
__device__ __forceinline__ int block_compact(const int32_t *__restrict__ v, int j0, int j1, int32_t thr, int run,
                                             int *warp_part, uint16_t *places, Emit emit)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int base = j0; base < j1; base += KEEP_ROUND) {
        const int w0 = base + warp * 256 + lane;
        int32_t x[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) x[u] = w0 + 32 * u < j1 ? v[w0 + 32 * u] : INT_MIN;
        unsigned mask[8];
        int found = 0;
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            mask[u] = __ballot_sync(0xffffffffu, w0 + 32 * u < j1 && x[u] >= thr);
            found += __popc(mask[u]);
        }
        int tot;
        int pos = sel_block_scan(lane == 0 ? found : 0, &tot, warp_part);       // (behind its barriers the last round's places are read)
        pos = __shfl_sync(0xffffffffu, pos, 0);
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            if (mask[u] >> lane & 1u) places[pos + __popc(mask[u] & ((1u << lane) - 1))] = (uint16_t)(w0 + 32 * u - base);
            pos += __popc(mask[u]);
        }
        __syncthreads();
        for (int i = threadIdx.x; i < tot; i += SEL_THREADS) emit(base + places[i], run + i);
        run += tot;
    }
    return run;
}
__device__ __forceinline__ void slice_of(int n, int *j0, int *j1)
{
    const int per = (n + (int)gridDim.x - 1) / (int)gridDim.x;
    *j0 = blockIdx.x * per < n ? blockIdx.x * per : n;
    *j1 = *j0 + per < n ? *j0 + per : n;
}
// Elements of the slices before this block's (counts[slice]; none when there is one slice).
__device__ __forceinline__ int slices_before(const int32_t *counts)
{
    int run = 0;
    for (int s = 0; s < (int)blockIdx.x; ++s) run += counts[s];
    return run;
}
// Elements of [j0, j1) with v >= thr (thr > INT_MIN).
__device__ __forceinline__ int block_count(const int32_t *__restrict__ v, int j0, int j1, int32_t thr, int *warp_part)
{
    int keep = 0;
    for (int base = j0; base < j1; base += 8 * SEL_THREADS) {
        int32_t x[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const int j = base + u * SEL_THREADS + threadIdx.x;
            x[u] = j < j1 ? v[j] : INT_MIN;
        }
#pragma unroll
        for (int u = 0; u < 8; ++u) keep += x[u] >= thr ? 1 : 0;
    }
    int total;
    sel_block_scan(keep, &total, warp_part);
    return total;
}

// grid (split, B).  tau = the n_prune-th largest exact CI of the seeds -> tau[b]; how many candidates of each slice have
// hi0 >= tau -> counts[b][slice].  Fewer seeds than n_prune (then there are few candidates): everything is kept.
__global__ void __launch_bounds__(SEL_THREADS)
filter_count_kernel(const int32_t *__restrict__ n_cand, const int32_t *__restrict__ hi0, int64_t maxc,
                    const int32_t *__restrict__ seed_ci, const int32_t *__restrict__ n_seed, int n_prune, int us,
                    int32_t *__restrict__ tau_out, int32_t *__restrict__ counts, int32_t *__restrict__ n_rest, FirstCut cut)
{
    pdl_entry();
    __shared__ int hist[2048];
    __shared__ int warp_part[32];
    __shared__ uint32_t s_prefix;
    __shared__ int s_want;
    const bool on = cut.on();
    const int b = blockIdx.y;
    int32_t tau = INT_MIN + 1;
    const int seeds = n_seed[b];
    if (!on) return;
    if (seeds >= n_prune) {
        const int32_t *sb = seed_ci + (int64_t)b * maxc;
        int need_eq;
        const uint32_t u = radix_select([&](int j) { return sb[j]; }, seeds, n_prune, hist, warp_part, &s_prefix,
                                        &s_want, &need_eq);
        tau = (int32_t)(u ^ 0x80000000u);
    }
    int j0, j1;
    slice_of(n_cand[b], &j0, &j1);
    const int total = block_count(hi0 + (int64_t)b * maxc, j0, j1, units_up(tau, us), warp_part);
    if (threadIdx.x == 0) {
        counts[(int64_t)b * KEEP_SPLIT + blockIdx.x] = total;
        if (blockIdx.x == 0) {
            tau_out[b] = tau;
            n_rest[b] = 0;                               // (counted up by the bounds of what is kept)
        }
    }
}

// Same grid: the kept candidates, ascending, behind those of the slices before, with their token ranges.  A seed's exact CI
// is known already: its range is (CI, 0), which the later kernels pass through.  Without the cut: all candidates.
__global__ void __launch_bounds__(SEL_THREADS)
filter_write_kernel(const int32_t *__restrict__ cand, const int32_t *__restrict__ n_cand,
                    const int64_t *__restrict__ doc_off, const int32_t *__restrict__ hi0, int64_t maxc,
                    const int32_t *__restrict__ seed_thr, const int32_t *__restrict__ seed_slot,
                    const int32_t *__restrict__ seed_ci, const int32_t *__restrict__ tau, int us,
                    const int32_t *__restrict__ counts, int32_t *__restrict__ kept, int2 *__restrict__ kept_rng,
                    int32_t *__restrict__ n_kept, FirstCut cut)
{
    pdl_entry();
    __shared__ int warp_part[32];
    __shared__ uint16_t places[KEEP_ROUND];
    const int b = blockIdx.y;
    const int64_t row = (int64_t)b * maxc;
    const bool on = cut.on();
    const int n = n_cand[b];
    int j0, j1;
    slice_of(n, &j0, &j1);
    if (!on) {
#pragma unroll 4
        for (int j = j0 + threadIdx.x; j < j1; j += SEL_THREADS) {
            const int32_t d = cand[row + j];
            kept[row + j] = d;
            kept_rng[row + j] = doc_range(doc_off, d);
        }
        if (blockIdx.x == 0 && threadIdx.x == 0) n_kept[b] = n;
        return;
    }
    const int32_t thr = seed_thr[b];
    const int run = block_compact(hi0 + row, j0, j1, units_up(tau[b], us), slices_before(counts + (int64_t)b * KEEP_SPLIT),
                                  warp_part, places, [&](int j, int pos) {
        const int32_t d = cand[row + j];
        kept[row + pos] = d;
        kept_rng[row + pos] = hi0[row + j] >= thr ? make_int2(seed_ci[row + seed_slot[row + j]], 0) : doc_range(doc_off, d);
    });
    if (blockIdx.x == gridDim.x - 1 && threadIdx.x == 0) n_kept[b] = run;
}

// What an upper bound has to reach: tau of the seeds, or without the cut the n_prune-th largest 8-bit lower bound.
__device__ __forceinline__ int32_t contend_threshold(const int32_t *lo, int n, int n_prune, int nq, int32_t tau, bool cut,
                                                     int *hist, int *warp_part, int *s_bin)
{
    if (cut) return tau;
    return n > n_prune ? contender_threshold(lo, n, n_prune, nq, hist, warp_part, s_bin) : INT_MIN + 1;
}

// grid (split, B): contenders = kept candidates whose 8-bit upper bound reaches the threshold, with their ranges, ascending.
// With several slices the count kernel runs first and leaves the threshold in tau.
__global__ void __launch_bounds__(SEL_THREADS)
filter_contend_count_kernel(const int32_t *__restrict__ n_kept, const int32_t *__restrict__ lo, const int32_t *__restrict__ hi,
                            int64_t maxc, int n_prune, int nq, const int32_t *tau_in, int32_t *tau_out,
                            int32_t *__restrict__ counts, FirstCut cut)
{
    pdl_entry();
    __shared__ int hist[CONT_BINS];
    __shared__ int warp_part[32];
    __shared__ int s_bin;
    const int b = blockIdx.y;
    const int64_t row = (int64_t)b * maxc;
    const bool on = cut.on();
    const int n = n_kept[b];
    const int32_t thr = contend_threshold(lo + row, n, n_prune, nq, tau_in[b], on, hist, warp_part, &s_bin);
    int j0, j1;
    slice_of(n, &j0, &j1);
    const int total = block_count(hi + row, j0, j1, thr, warp_part);
    if (threadIdx.x == 0) {
        counts[(int64_t)b * KEEP_SPLIT + blockIdx.x] = total;
        if (blockIdx.x == 0 && !on) tau_out[b] = thr;
    }
}
__global__ void __launch_bounds__(SEL_THREADS)
filter_contend_kernel(const int32_t *__restrict__ kept, const int2 *__restrict__ kept_rng, const int32_t *__restrict__ n_kept,
                      const int32_t *__restrict__ lo, const int32_t *__restrict__ hi, int64_t maxc, int n_prune, int nq,
                      const int32_t *__restrict__ tau, const int32_t *__restrict__ counts, int32_t *__restrict__ cont,
                      int2 *__restrict__ cont_rng, int32_t *__restrict__ n_cont, FirstCut cut)
{
    pdl_entry();
    __shared__ int hist[CONT_BINS];
    __shared__ int warp_part[32];
    __shared__ int s_bin;
    const int b = blockIdx.y;
    const int64_t row = (int64_t)b * maxc;
    const bool known = cut.on() || gridDim.x > 1;       // (the threshold is in tau)
    const int n = n_kept[b];
    const int32_t thr = contend_threshold(lo + row, n, n_prune, nq, tau[b], known, hist, warp_part, &s_bin);
    int j0, j1;
    slice_of(n, &j0, &j1);
    uint16_t *places = reinterpret_cast<uint16_t *>(hist);  // (read before the first of the scan's barriers, if at all)
    const int run = block_compact(hi + row, j0, j1, thr, slices_before(counts + (int64_t)b * KEEP_SPLIT), warp_part,
                                  places, [&](int j, int pos) {
        cont[row + pos] = kept[row + j];
        cont_rng[row + pos] = kept_rng[row + j];
    });
    if (blockIdx.x == gridDim.x - 1 && threadIdx.x == 0) n_cont[b] = run;
}

// ------------------------------------------------------------------------------------------------ launchers -------
// Units of e and hi0: 2^us.  2^16 from the 8-bit table and for the 6-bit codes; the exact table gives finer ones, as fine as
// 16 bits hold for q_len columns.
static int filter_unit(const Index &ix, const Params &p, bool from_table8)
{
    return from_table8 || filter_codec(ix.K) != 16 ? 16 : p.nq <= 63 ? 14 : 15;
}

// The scan a query at a time.
static int launch_query_scan(const Index &ix, const Params &p, const Layout &L, const int32_t *table, uint8_t *table8, int us,
                             const int32_t *cand, const int32_t *n_cand, int32_t *hi0, char *ws, cudaStream_t st)
{
    int32_t *theta = (int32_t *)(ws + L.flt_theta), *hist = (int32_t *)(ws + L.flt_hist);
    const FirstCut cut = first_cut(p, L, ws);
    uint8_t *tab = (uint8_t *)(ws + L.flt_tab);
    uint32_t *mask = (uint32_t *)(ws + L.flt_mask);
    const bool ready = coarse_supported(p.nq);           // stage 1 has written the 8-bit table
    const int codec = filter_codec(ix.K);
    const size_t pitch = filter_table_pitch(ix);
    int64_t gx = (8LL * ix.sm_count + p.B - 1) / p.B;
    if (ready) {
        const int64_t want = ((codec == 16 ? ix.K : (ix.K + 4) / 5) + 255) / 256;
        if (gx > want) gx = want;
        const dim3 grid((unsigned)gx, (unsigned)p.B);
        if (p.nq == 32 && codec == 16) launch(filter_excess_kernel<8, 16>, grid, 256, 0, st, table8, ix.K, theta, tab, pitch, mask, cut);
        else if (p.nq == 32) launch(filter_excess_kernel<8, 6>, grid, 256, 0, st, table8, ix.K, theta, tab, pitch, mask, cut);
        else if (codec == 16) launch(filter_excess_kernel<16, 16>, grid, 256, 0, st, table8, ix.K, theta, tab, pitch, mask, cut);
        else launch(filter_excess_kernel<16, 6>, grid, 256, 0, st, table8, ix.K, theta, tab, pitch, mask, cut);
    } else {
        const int64_t want = (ix.K + 39) / 40;
        if (gx > want) gx = want;
        const dim3 grid((unsigned)gx, (unsigned)p.B);
        auto kern = codec == 16 ? (p.nq <= 32   ? filter_excess_exact_kernel<16, 1>
                                   : p.nq <= 64 ? filter_excess_exact_kernel<16, 2>
                                                : filter_excess_exact_kernel<16, 4>)
                                : (p.nq <= 32   ? filter_excess_exact_kernel<6, 1>
                                   : p.nq <= 64 ? filter_excess_exact_kernel<6, 2>
                                                : filter_excess_exact_kernel<6, 4>);
        launch(kern, grid, 256, 0, st, table, ix.K, p.nq, theta, us, table8, tab, pitch, (uint8_t *)mask);
    }
    CHIMERA_CUDA(cudaGetLastError());

    // Blocks per query: one block is resident per SM.  About eight waves over the batch even out the queries; few blocks
    // per query keep many queries in step over the same documents, whose centroid ids then come from L2.
    gx = (8LL * ix.sm_count + p.B - 1) / p.B;
    if (gx > ix.sm_count) gx = ix.sm_count;
    const int64_t want = (p.maxc + 511) / 512;
    if (gx > want) gx = want;
    const dim3 grid((unsigned)gx, (unsigned)p.B);
    if (codec == 16) {
        CHIMERA_CUDA(allow_shared(filter_scan_kernel<16>, FILTER_SMEM));
        launch(filter_scan_kernel<16>, grid, SCAN_THREADS_F, pitch, st, tab, pitch, theta, p.nq, us, cand, ix.doc_off, n_cand, p.maxc,
                                                                    ix.cids, ix.T, hi0, hist, cut);
    } else {
        CHIMERA_CUDA(allow_shared(filter_scan_kernel<6>, FILTER_SMEM));
        launch(filter_scan_kernel<6>, grid, SCAN_THREADS_F, pitch, st, tab, pitch, theta, p.nq, us, cand, ix.doc_off, n_cand, p.maxc,
                                                                   ix.cids, ix.T, hi0, hist, cut);
    }
    CHIMERA_CUDA(cudaGetLastError());
    count_launch(SLOT_CI, 2);
    return CHIMERA_OK;
}

int launch_filter_scan(const Index &ix, const Params &p, const Layout &L, bool batch, const int32_t *table, uint8_t *table8,
                       const int32_t *cand, const int32_t *n_cand, int32_t *hi0, int32_t *seed,
                       int2 *seed_rng, char *ws, cudaStream_t st)
{
    int32_t *theta = (int32_t *)(ws + L.flt_theta), *hist = (int32_t *)(ws + L.flt_hist);
    int32_t *n_seed = (int32_t *)(ws + L.n_seed), *vote = (int32_t *)(ws + L.flt_vote);
    const FirstCut cut = first_cut(p, L, ws);
    const bool ready = coarse_supported(p.nq);           // stage 1 has written the 8-bit table
    const int codec = filter_codec(ix.K);
    const int step = (int)(ix.K / FILTER_SAMPLE > 1 ? ix.K / FILTER_SAMPLE : 1);
    const int m = (int)((ix.K + step - 1) / step < 2 * FILTER_SAMPLE ? (ix.K + step - 1) / step : 2 * FILTER_SAMPLE);
    int rank = (int)(filter_share(ix) * m + 0.5);
    if (rank < 1) rank = 1;
    const unsigned groups = (unsigned)((p.nq + 31) / 32);
    const int parts = filter_parts(ix, p);
    int32_t *parts_hist = (int32_t *)(ws + L.flt_parts), *done = parts_hist + (size_t)p.B * groups * 256 * 32;
    if (parts > 1)
        CHIMERA_CUDA(cudaMemsetAsync(parts_hist, 0, filter_parts_bytes(ix, p), st));
    const dim3 grid(groups, (unsigned)p.B, (unsigned)parts);
    if (ready)
        launch(filter_theta_kernel<uint8_t>, grid, SEL_THREADS, 0, st, (const uint8_t *)table8, ix.K, p.nq, m, step, rank, theta, hist, n_seed,
               parts_hist, done, vote);
    else
        launch(filter_theta_kernel<int32_t>, grid, SEL_THREADS, 0, st, table, ix.K, p.nq, m, step, rank, theta, hist, n_seed, parts_hist, done,
               (int32_t *)nullptr);
    CHIMERA_CUDA(cudaGetLastError());
    const int us = filter_unit(ix, p, ready);
    int rc;
    if (batch && (rc = launch_batch_quantum(ix, p, L, table, table8, us, ws, st))) return rc;
    if (ready) {
        const int jq = cut_queries(p);
        const dim3 grid((unsigned)(cut_samples(p) / 32), (unsigned)jq);
        launch(p.nq == 32 ? filter_sample_kernel<32> : filter_sample_kernel<64>, grid, SEL_THREADS, 0, st, table8, ix.K, theta, p.B,
               cand, n_cand, p.maxc, ix.doc_off, ix.cids, p.n_prune, codec == 6, batch ? (const int2 *)(ws + L.flt_over) : nullptr,
               (int2 *)(ws + L.flt_smp), vote);
        CHIMERA_CUDA(cudaGetLastError());
        count_launch(SLOT_CI);
    }

    if (batch) {
        if ((rc = launch_batch_scan(ix, p, L, table, table8, us, n_cand, hi0, ws, st))) return rc;
    } else if ((rc = launch_query_scan(ix, p, L, table, table8, us, cand, n_cand, hi0, ws, st))) {
        return rc;
    }
    // 2 n_prune for q_len 32 / 64, whose exact rows are read in 16-byte pieces (Mid, batch 256: 1.5 n_prune 6,641 us, 2 6,419, 2.5
    // 6,437), 1.5 n_prune for others, where an exact row costs three to four times its 8-bit copy (37 queries of 21 tokens: 1.5
    // 1,047 us, 2.5 1,148)
    launch(filter_seed_kernel, dim3((unsigned)filter_split(ix, p), (unsigned)p.B), SEL_THREADS, 0, st, cand, n_cand, ix.doc_off, hi0, p.maxc, theta, p.nq, us, hist, (ready ? 2 * p.n_prune : p.n_prune + p.n_prune / 2) + 32, seed, seed_rng, n_seed,
        (int32_t *)(ws + L.flt_thr), (int32_t *)(ws + L.flt_slot), cut);
    CHIMERA_CUDA(cudaGetLastError());
    count_launch(SLOT_CI, 2);                            // (with the thresholds)
    return CHIMERA_OK;
}

int launch_filter_keep(const Index &ix, const Params &p, const Layout &L, const int32_t *cand,
                       const int32_t *n_cand, const int32_t *hi0, const int32_t *seed_ci, int32_t *kept,
                       int2 *kept_rng, int32_t *n_kept, char *ws, cudaStream_t st)
{
    const int32_t *n_seed = (const int32_t *)(ws + L.n_seed);
    int32_t *counts = (int32_t *)(ws + L.flt_counts);
    const int us = filter_unit(ix, p, coarse_supported(p.nq));
    int32_t *tau = (int32_t *)(ws + L.flt_tau);
    const FirstCut cut = first_cut(p, L, ws);
    const int32_t *thr = (const int32_t *)(ws + L.flt_thr), *slot = (const int32_t *)(ws + L.flt_slot);
    const dim3 grid((unsigned)filter_split(ix, p), (unsigned)p.B);
    launch(filter_count_kernel, grid, SEL_THREADS, 0, st, n_cand, hi0, p.maxc, seed_ci, n_seed, p.n_prune, us, tau, counts,
           (int32_t *)(ws + L.n_rest), cut);
    CHIMERA_CUDA(cudaGetLastError());
    launch(filter_write_kernel, grid, SEL_THREADS, 0, st, cand, n_cand, ix.doc_off, hi0, p.maxc, thr, slot, seed_ci, tau, us,
                                                      counts, kept, kept_rng, n_kept, cut);
    CHIMERA_CUDA(cudaGetLastError());
    count_launch(SLOT_SELECT, 2);
    return CHIMERA_OK;
}

int launch_filter_contenders(const Index &ix, const Params &p, const Layout &L, const int32_t *kept, const int2 *kept_rng,
                             const int32_t *n_kept, const int32_t *lo, const int32_t *hi, int32_t *cont, int2 *cont_rng,
                             int32_t *n_cont, char *ws, cudaStream_t st)
{
    int32_t *counts = (int32_t *)(ws + L.flt_counts), *tau = (int32_t *)(ws + L.flt_tau);
    const FirstCut cut = first_cut(p, L, ws);
    // one block per query keeps up in a large batch; a single query's list is spread
    const int split = 4 * p.B <= ix.sm_count ? filter_split(ix, p) : 1;
    const dim3 grid((unsigned)split, (unsigned)p.B);
    if (split > 1) {
        launch(filter_contend_count_kernel, grid, SEL_THREADS, 0, st, n_kept, lo, hi, p.maxc, p.n_prune, p.nq, tau, tau, counts, cut);
        CHIMERA_CUDA(cudaGetLastError());
        count_launch(SLOT_SELECT);
    }
    launch(filter_contend_kernel, grid, SEL_THREADS, 0, st, kept, kept_rng, n_kept, lo, hi, p.maxc, p.n_prune, p.nq, tau, counts,
           cont, cont_rng, n_cont, cut);
    CHIMERA_CUDA(cudaGetLastError());
    count_launch(SLOT_SELECT);
    return CHIMERA_OK;
}

}  // namespace chimera
