// Stage 2b: candidate documents of a query = every document that owns a token in one of the probed posting lists
// (Sec. 3.2 step 1: L_q is the union of the probed lists, S the set of their source documents).
//
// The inverted file stores, per centroid, the unique ids of those documents.  Each probed list is streamed once and
// sets one bit per document in a per-query bitmap (the dedup); the bitmap is then compacted into an ascending id list with
// the documents' token ranges: a count per chunk of the bitmap and an ordered write, or, for few queries on small corpora, the
// write alone over shorter chunks, each of which counts the words before its own.
#include "common.cuh"

namespace chimera {

// grid (nq * P, B): one block per probed list.
__global__ void __launch_bounds__(128)
mark_kernel(const int32_t *__restrict__ probes, int n_lists, const int64_t *__restrict__ ivf_off,
            const int32_t *__restrict__ ivf_doc, uint32_t *__restrict__ bitmap, int64_t words)
{
    pdl_entry();
    const int b = blockIdx.y;
    const int32_t c = DBG_CID(probes[(int64_t)b * n_lists + blockIdx.x]);
    uint32_t *bm = bitmap + (int64_t)b * words;
    const int64_t lo = ivf_off[c], hi = ivf_off[c + 1];
    // four list entries per thread and iteration: their loads and the bitmap reads they lead to are in flight together
    for (int64_t e0 = lo + threadIdx.x; e0 < hi; e0 += 4 * (int64_t)blockDim.x) {
        uint32_t d[4], cur[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int64_t e = e0 + u * (int64_t)blockDim.x;
            d[u] = e < hi ? (uint32_t)ivf_doc[e] : 0xffffffffu;
            if (e < hi && !DBG_DOC_OK(d[u])) d[u] = 0xffffffffu;          // (debug build) skip a bad list entry
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) cur[u] = d[u] != 0xffffffffu ? bm[d[u] >> 5] : 0xffffffffu;
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const uint32_t bit = 1u << (d[u] & 31);
            if (!(cur[u] & bit)) atomicOr(&bm[d[u] >> 5], bit);
        }
    }
}

// The same with the bitmap in shared memory, for small corpora: their lists set the same few words over and over, and
// atomics on one L2 line come one after the other (10,000 documents, 128 lists of 625: 17 us, here 6.5).  grid (blocks, B): a
// block takes every gridDim.x-th list and adds its bits to the query's bitmap at the end.  Its warps take the lists in
// pieces of 256 entries (a warp per list, the longest one took the time: one query, 400,000 documents, 1,024 lists
// of popular centroids, stage 2b 189 us in 16 blocks, 112 so and 70 in 32).
constexpr int MARK_SHARED_WORDS = 24 * 1024;
__global__ void __launch_bounds__(512)
mark_shared_kernel(const int32_t *__restrict__ probes, int n_lists, const int64_t *__restrict__ ivf_off,
                   const int32_t *__restrict__ ivf_doc, uint32_t *__restrict__ bitmap, int words)
{
    pdl_entry();
    extern __shared__ uint32_t bits[];
    const int b = blockIdx.y;
    for (int w = threadIdx.x; w < words; w += 512) bits[w] = 0u;
    __syncthreads();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int l0 = blockIdx.x; l0 < n_lists; l0 += 32 * gridDim.x) {
        const int l = l0 + lane * (int)gridDim.x;
        int64_t lo = 0;                                      // of this lane's list
        int len = 0;
        if (l < n_lists) {
            const int32_t c = DBG_CID(probes[(int64_t)b * n_lists + l]);
            lo = ivf_off[c];
            len = (int)(ivf_off[c + 1] - lo);
        }
        const int pieces = (len + 255) >> 8;
        int end = pieces;                                    // of this list's pieces among those of the 32
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int t = __shfl_up_sync(0xffffffffu, end, o);
            if (lane >= o) end += t;
        }
        const int all = __shfl_sync(0xffffffffu, end, 31);
        for (int piece = warp; piece < all; piece += 16) {
            const int i = __ffs(__ballot_sync(0xffffffffu, end > piece)) - 1;
            const int from = 256 * (piece - __shfl_sync(0xffffffffu, end - pieces, i)) + lane;
            const int left = __shfl_sync(0xffffffffu, len, i) - from;
            const int32_t *src = ivf_doc + __shfl_sync(0xffffffffu, lo, i) + from;
            uint32_t d[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                d[u] = 32 * u < left ? (uint32_t)src[32 * u] : 0xffffffffu;
                if (d[u] != 0xffffffffu && !DBG_DOC_OK(d[u])) d[u] = 0xffffffffu;
            }
#pragma unroll
            for (int u = 0; u < 8; ++u)
                if (d[u] != 0xffffffffu) {
                    const uint32_t bit = 1u << (d[u] & 31);
                    if (!(bits[d[u] >> 5] & bit)) atomicOr(&bits[d[u] >> 5], bit);
                }
            __syncwarp();
        }
    }
    __syncthreads();
    for (int w = threadIdx.x; w < words; w += 512)
        if (bits[w]) atomicOr(&bitmap[(int64_t)b * words + w], bits[w]);
}

// Large batches: a block owns a range of a query's bitmap in shared memory, reads all of the query's lists and keeps the
// documents of its range (a list is not sorted, and re-reading it from L2 is cheaper than an atomic in L2 per entry); the
// range is stored once, so nothing is cleared before, and its chunks are counted on the way.  grid (ranges, B).
// Measured (batch 256, marking and counting): Mid, one range of 62 KB: 233 -> 36 us; Large, five of 220 KB: 850 -> 347 us.
constexpr int MARK_RANGE_WORDS = 55 * 1024;              // 220 KB of shared memory, whole chunks
__global__ void __launch_bounds__(1024)
mark_range_kernel(const int32_t *__restrict__ probes, int n_lists, const int64_t *__restrict__ ivf_off,
                  const int32_t *__restrict__ ivf_doc, uint32_t *__restrict__ bitmap, int64_t words, int range_words,
                  int n_chunks, int32_t *__restrict__ chunk_cnt)
{
    pdl_entry();
    extern __shared__ uint32_t bits[];
    const int b = blockIdx.y, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t first = (int64_t)blockIdx.x * range_words;
    const int n = (int)(words - first < range_words ? words - first : range_words);
    for (int w = threadIdx.x; w < range_words; w += 1024) bits[w] = 0u;
    __syncthreads();
    const uint32_t doc0 = (uint32_t)(first << 5), docs = (uint32_t)n << 5;
    for (int l = warp; l < n_lists; l += 32) {
        const int32_t c = DBG_CID(probes[(int64_t)b * n_lists + l]);
        const int64_t hi = ivf_off[c + 1];
        for (int64_t e0 = ivf_off[c] + lane; e0 < hi; e0 += 8 * 32) {
            uint32_t d[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                d[u] = e0 + 32 * u < hi ? (uint32_t)__ldg(ivf_doc + e0 + 32 * u) : 0xffffffffu;
                if (d[u] != 0xffffffffu && !DBG_DOC_OK(d[u])) d[u] = 0xffffffffu;
                d[u] -= doc0;                            // (an entry of another range, and the filler, end up past `docs`)
            }
#pragma unroll
            for (int u = 0; u < 8; ++u)
                if (d[u] < docs) atomicOr(&bits[d[u] >> 5], 1u << (d[u] & 31));
        }
    }
    __syncthreads();
    for (int w = threadIdx.x; w < n; w += 1024) bitmap[(int64_t)b * words + first + w] = bits[w];
    // a warp per chunk
    for (int k = warp; k * BITMAP_CHUNK_WORDS < n; k += 32) {
        int c = 0;
#pragma unroll 8
        for (int w = lane; w < BITMAP_CHUNK_WORDS; w += 32) c += __popc(bits[k * BITMAP_CHUNK_WORDS + w]);
        c = __reduce_add_sync(0xffffffffu, c);
        if (lane == 0) chunk_cnt[(int64_t)b * n_chunks + first / BITMAP_CHUNK_WORDS + k] = c;
    }
}

constexpr int CHUNK_THREADS = 256;
constexpr int WORDS_PER_THREAD = BITMAP_CHUNK_WORDS / CHUNK_THREADS;   // at most: 4 consecutive words per thread
constexpr int COMPACT_STAGE = 8192;      // ids a chunk stages in shared memory (a chunk covers 32,768 documents)

__device__ __forceinline__ int block_exclusive_scan_256(int v, int *total)
{
    __shared__ int warp_part[CHUNK_THREADS / 32];
    int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int incl = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        int t = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += t;
    }
    if (lane == 31) warp_part[warp] = incl;
    __syncthreads();
    int before = 0, all = 0;
#pragma unroll
    for (int w = 0; w < CHUNK_THREADS / 32; ++w) {
        int pw = warp_part[w];
        if (w < warp) before += pw;
        all += pw;
    }
    *total = all;
    return before + incl - v;
}

// grid (n_chunks, B): number of set bits in each chunk -> chunk_cnt[b][chunk].
__global__ void __launch_bounds__(CHUNK_THREADS)
count_kernel(const uint32_t *__restrict__ bitmap, int64_t words, int n_chunks, int32_t *__restrict__ chunk_cnt)
{
    pdl_entry();
    const int b = blockIdx.y;
    const uint32_t *bm = bitmap + (int64_t)b * words;
    int64_t w0 = (int64_t)blockIdx.x * BITMAP_CHUNK_WORDS + threadIdx.x * WORDS_PER_THREAD;
    int c = 0;
#pragma unroll
    for (int j = 0; j < WORDS_PER_THREAD; ++j)
        if (w0 + j < words) c += __popc(bm[w0 + j]);
    int total;
    block_exclusive_scan_256(c, &total);
    if (threadIdx.x == 0) chunk_cnt[(int64_t)b * n_chunks + blockIdx.x] = total;
}

// grid (n_chunks, B): write the ids of the set bits of each chunk, ascending, behind those of the chunks before it (whose
// counts are in chunk_cnt; NULL: their words are counted here), and the documents' token ranges (rng may be NULL).  The last
// chunk's block reports the query's candidates (clamped to maxc; an overflow sets the status bit).  cont_hist (may be NULL):
// scratch rows whose first `hist_n` entries are cleared for a later kernel.
__global__ void __launch_bounds__(CHUNK_THREADS)
compact_kernel(const uint32_t *__restrict__ bitmap, int64_t words, int n_chunks, int chunk_words,
               const int32_t *__restrict__ chunk_cnt, int64_t maxc, int32_t *__restrict__ cand,
               int32_t *__restrict__ n_cand, uint2 *__restrict__ ranks, const int64_t *__restrict__ doc_off,
               int2 *__restrict__ rng, int32_t *__restrict__ cont_hist, int hist_n, uint32_t *status)
{
    pdl_entry();
    __shared__ int s_base;
    if (threadIdx.x == 0) s_base = 0;
    if (cont_hist)
        for (int i = blockIdx.x * CHUNK_THREADS + threadIdx.x; i < hist_n; i += gridDim.x * CHUNK_THREADS)
            cont_hist[(int64_t)blockIdx.y * maxc + i] = 0;
    __syncthreads();
    {
        int before = 0;
        if (chunk_cnt) {
            for (int c = threadIdx.x; c < (int)blockIdx.x; c += CHUNK_THREADS)
                before += chunk_cnt[(int64_t)blockIdx.y * n_chunks + c];
        } else {
            const uint32_t *bm = bitmap + (int64_t)blockIdx.y * words;
            const int n = (int)blockIdx.x * chunk_words;
#pragma unroll 8
            for (int w = threadIdx.x; w < n; w += CHUNK_THREADS) before += __popc(bm[w]);
        }
        before = __reduce_add_sync(0xffffffffu, before);
        if ((threadIdx.x & 31) == 0 && before) atomicAdd(&s_base, before);
    }
    const int b = blockIdx.y;
    const uint32_t *bm = bitmap + (int64_t)b * words;
    const int wpt = chunk_words > CHUNK_THREADS ? chunk_words / CHUNK_THREADS : 1;
    const int64_t w0 = (int64_t)blockIdx.x * chunk_words + threadIdx.x * wpt;
    const int mine = (int)threadIdx.x * wpt < chunk_words ? wpt : 0;      // words of this thread
    uint32_t w[WORDS_PER_THREAD];
    int c = 0;
#pragma unroll
    for (int j = 0; j < WORDS_PER_THREAD; ++j) {
        w[j] = (j < mine && w0 + j < words) ? bm[w0 + j] : 0u;
        c += __popc(w[j]);
    }
    int total;
    const int local = block_exclusive_scan_256(c, &total);      // (its barrier is also the one behind s_base)
    const int64_t base = s_base;
    if (threadIdx.x == 0 && (int)blockIdx.x == n_chunks - 1) {
        const int64_t all = base + total;
        if (all > maxc) atomicOr(status, ST_OVERFLOW);
        n_cand[b] = (int32_t)(all < maxc ? all : maxc);
    }
    int32_t *out = cand + (int64_t)b * maxc;
    // A thread's ids are consecutive in the output but the threads' runs are ~30 ids apart, so direct stores are
    // scattered 4-byte writes: when the chunk's ids fit, they are staged in shared memory and copied out coalesced.  A fuller chunk
    // (a quarter of its documents) is written a bitmap word per warp, from the words and the positions that they start at (64
    // queries with all of 200,000 documents: 117 -> 24 us).
    __shared__ __align__(8) int32_t staged[COMPACT_STAGE];
    uint2 *starts = reinterpret_cast<uint2 *>(staged);
    static_assert(sizeof(uint2) * BITMAP_CHUNK_WORDS <= sizeof(staged), "words and positions of a chunk");
    const bool use_stage = total <= COMPACT_STAGE;
    int64_t pos = use_stage ? local : base + local;
#pragma unroll
    for (int j = 0; j < WORDS_PER_THREAD; ++j) {
        uint32_t bits = w[j];
        if (ranks && j < mine && w0 + j < words)          // the word and the candidates before it: document -> candidate index
            ranks[(int64_t)b * words + w0 + j] = make_uint2(w[j], (uint32_t)(use_stage ? base + pos : pos));
        if (!use_stage) {
            if (j < mine) starts[threadIdx.x * wpt + j] = make_uint2(w[j], (uint32_t)pos);
            pos += __popc(bits);
            continue;
        }
        while (bits) {
            int t = __ffs(bits) - 1;
            bits &= bits - 1;
            staged[pos++] = (int32_t)(((w0 + j) << 5) + t);
        }
    }
    if (!use_stage) {
        __syncthreads();
        const int lane = threadIdx.x & 31;
        constexpr int W = 4;                                 // words in flight
        for (int i0 = threadIdx.x >> 5; i0 < chunk_words; i0 += W * (CHUNK_THREADS / 32)) {
            int64_t at[W];
            int32_t id[W];
#pragma unroll
            for (int u = 0; u < W; ++u) {
                const int i = i0 + u * (CHUNK_THREADS / 32);
                const uint2 s = i < chunk_words ? starts[i] : make_uint2(0u, 0u);
                at[u] = s.x >> lane & 1u ? (int64_t)s.y + __popc(s.x & ((1u << lane) - 1u)) : maxc;
                id[u] = (int32_t)((((int64_t)blockIdx.x * chunk_words + i) << 5) + lane);
            }
#pragma unroll
            for (int u = 0; u < W; ++u)
                if (at[u] < maxc) out[at[u]] = id[u];
            if (rng) {
                int2 r[W];
#pragma unroll
                for (int u = 0; u < W; ++u) r[u] = at[u] < maxc ? doc_range(doc_off, id[u]) : make_int2(0, 0);
#pragma unroll
                for (int u = 0; u < W; ++u)
                    if (at[u] < maxc) rng[(int64_t)b * maxc + at[u]] = r[u];
            }
        }
        return;
    }
    __syncthreads();
    for (int e = threadIdx.x; e < total; e += CHUNK_THREADS)
        if (base + e < maxc) {
            out[base + e] = staged[e];
            if (rng) rng[(int64_t)b * maxc + base + e] = doc_range(doc_off, staged[e]);
        }
}

// In shared memory: bitmaps of up to 96 KB whose words are set a dozen times or more on average.  By range: a block per query and
// range (every range reads all lists: up to 14 million documents), for more queries than a quarter of the SMs, unless that leaves half
// of them idle and the lists are long enough for sixteen blocks.  In L2: the others.
// Measured (stage 2b in us, means over 8,000 to 760,000 documents, lists of 300 to 6,000, even and popular centroids, 32 to 1,024 lists; in
// L2 / in shared memory / by range):
//   by times that a word is set, 1 query: 6 to 12 times 25 / 22, 12 to 24 29 / 24, more than 100 51 / 25; 4 queries 25 / 19, 40 / 24, 71 / 26;
//     37: 69 / 42, 138 / 72, 247 / 65.  Set fewer times, even lists are as fast in L2, and a little faster with one query.
//   by queries, 24 times or more: 48 246 / 79 / 124; 64 305 / 89 / 126; 96 361 / 101 / 108; 128 457 / 122 / 111.  Even lists alone: 64 queries
//     of 128 lists of 300, 50,000 documents 40 / 31 / 28; 96 queries of 1,024 lists, 8,000 documents 561 / 85 / 61.
int gather_form(const Index &ix, const Params &p)
{
    const int64_t words = (ix.N + 31) / 32, ranges = (words + MARK_RANGE_WORDS - 1) / MARK_RANGE_WORDS;
    const double entries = (double)p.nq * p.P * ((double)ix.ivf_len / (double)ix.K);
    const bool shared = words <= MARK_SHARED_WORDS && entries >= 12.0 * (double)words;
    if (4 * p.B > ix.sm_count && ranges <= 8 && !(shared && 2 * ranges * p.B <= ix.sm_count && entries >= 65536.0)) return GATHER_RANGES;
    return shared ? GATHER_SHARED : GATHER_L2;
}

int launch_gather(const Index &ix, const Params &p, const Layout &L, const int32_t *probes, uint32_t *bitmap,
                  bool bitmap_clear, int32_t *chunk_cnt, int32_t *cand, int32_t *n_cand, uint2 *ranks, int2 *rng,
                  int32_t *cont_scratch, uint32_t *status, cudaStream_t st)
{
    const int n_lists = p.nq * p.P;
    const bool few = 4 * p.B <= ix.sm_count;
    const int ranges = (int)((L.words + MARK_RANGE_WORDS - 1) / MARK_RANGE_WORDS), form = gather_form(ix, p);
    const bool by_range = form == GATHER_RANGES;
    if (!by_range && !bitmap_clear) CHIMERA_CUDA(cudaMemsetAsync(bitmap, 0, sizeof(uint32_t) * (size_t)L.words * p.B, st));
    if (by_range) {
        int range_words = (int)((L.words + ranges - 1) / ranges);
        range_words = (range_words + BITMAP_CHUNK_WORDS - 1) / BITMAP_CHUNK_WORDS * BITMAP_CHUNK_WORDS;
        const size_t smem = sizeof(uint32_t) * (size_t)range_words;
        CHIMERA_CUDA(allow_shared(mark_range_kernel, sizeof(uint32_t) * MARK_RANGE_WORDS));
        launch(mark_range_kernel, dim3((unsigned)((L.words + range_words - 1) / range_words), (unsigned)p.B), 1024, smem, st, probes,
               n_lists, ix.ivf_off, ix.ivf_doc, bitmap, L.words, range_words, L.n_chunks, chunk_cnt);
    } else if (form == GATHER_SHARED) {
        // (32 blocks instead of 16, words set 24 times or more as above: one query 23 us instead of 29, eight 29 and 33, 16 39 and 39)
        const int blocks = p.B <= 8 ? 32 : 16;
        CHIMERA_CUDA(allow_shared(mark_shared_kernel, sizeof(uint32_t) * MARK_SHARED_WORDS));
        launch(mark_shared_kernel, dim3((unsigned)(n_lists < blocks ? n_lists : blocks), (unsigned)p.B), 512,
               sizeof(uint32_t) * (size_t)L.words, st, probes, n_lists, ix.ivf_off, ix.ivf_doc, bitmap, (int)L.words);
    } else {
        launch(mark_kernel, dim3((unsigned)n_lists, (unsigned)p.B), 128, 0, st, probes, n_lists, ix.ivf_off, ix.ivf_doc,
               bitmap, L.words);
    }
    CHIMERA_CUDA(cudaGetLastError());
    const dim3 gc((unsigned)L.n_chunks, (unsigned)p.B);
    // few queries on up to half a million documents: one launch of many short chunks, which count the words before them
    const bool one_pass = few && L.words <= 16 * 1024;
    constexpr int SHORT_CHUNK = 64;
    const dim3 gs((unsigned)((L.words + SHORT_CHUNK - 1) / SHORT_CHUNK), (unsigned)p.B);
    if (!one_pass && !by_range) {
        launch(count_kernel, gc, CHUNK_THREADS, 0, st, bitmap, L.words, L.n_chunks, chunk_cnt);
        CHIMERA_CUDA(cudaGetLastError());
    }
    launch(compact_kernel, one_pass ? gs : gc, CHUNK_THREADS, 0, st, bitmap, L.words, one_pass ? (int)gs.x : L.n_chunks,
           one_pass ? SHORT_CHUNK : BITMAP_CHUNK_WORDS, one_pass ? nullptr : chunk_cnt, p.maxc, cand,
           n_cand, ranks, ix.doc_off, rng, cont_scratch, contender_hist_entries(), status);
    CHIMERA_CUDA(cudaGetLastError());
    count_launch(SLOT_GATHER, one_pass || by_range ? 2 : 3);
    return CHIMERA_OK;
}

}  // namespace chimera
