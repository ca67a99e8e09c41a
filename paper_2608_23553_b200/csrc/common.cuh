// Shared declarations of libchimera's translation units (host side + small device helpers).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>
#include <stddef.h>

#include "chimera.h"

namespace chimera {

// ---------------------------------------------------------------------------------------------------------------
// Index: everything resident on the device between searches.
// ---------------------------------------------------------------------------------------------------------------
// Memory of copies in list order: an allocation of their own, or room behind the token lists.  Kept once it is there (the
// sizes of an index do not change).
struct ListMemory {
    void *at = nullptr;
    bool own = false;
};
struct Index {
    int device = 0;
    int sm_count = 0;
    int D = 0, nbits = 0, CB = 0;     // dim, residual bits per dim, code bytes per token
    int64_t K = 0, N = 0, T = 0;
    float res_lo = 0.f, res_hi = 0.f;
    const int32_t *cids = nullptr;    // [T]        borrowed
    const uint8_t *codes = nullptr;   // [T, CB]    borrowed
    int64_t *doc_off = nullptr;       // [N+1]      owned: first token of each document
    int8_t *cdig = nullptr;           // [3][K][128] owned: balanced base-256 digits of rint(c * 2^22), zero padded, digit_dim() order
    int64_t *ivf_off = nullptr;       // [K+1]      owned
    int32_t *ivf_doc = nullptr;       // [ivf_len]  owned: unique document ids per centroid, unordered
    int64_t ivf_len = 0;
    int32_t max_doclen = 0;
    // token-level posting lists (only after chimera_index_enable_partial): per centroid its tokens and their documents
    int64_t *tok_off = nullptr;       // [K+1]      owned, with the next two in the same allocation
    int32_t *tok_id = nullptr;        // [T]        token ids per centroid, unordered
    int32_t *tok_doc = nullptr;       // [T]        document of each listed token
    int64_t max_tok_list = 0;         // longest token list
    ListMemory code_mem, rq_mem;      // owned: the next one, the two behind it
    uint8_t *list_codes = nullptr;    // [T, CB]    optional: the codes in list order (see build_lists_and_copies)
    uint8_t *list_bits = nullptr;     // [T, D/8]   optional: the RaBitQ codes in list order
    float *list_inv = nullptr;        // [T]        their factors: both or neither
    // RaBitQ 1-bit codes (only after chimera_index_attach_rabitq)
    const uint8_t *rq_bits = nullptr; // [T, D/8]   borrowed: sign bits of the rotated tokens
    const float *rq_inv = nullptr;    // [T]        borrowed: 1 / <o_p, o_p-bar>
    float *rot_t = nullptr;           // [D][D]     owned: transposed rotation, rot_t[x * D + r] = P[r][x]
    // proximity graph over the centroids (only after chimera_index_build_graph)
    int32_t *graph = nullptr;         // [K][graph_deg] owned: nearest other centroids of each centroid, best first
    int32_t *xc = nullptr;            // [K][D]     owned: rint(centroid * 2^22)
    int graph_deg = 0;
};

// Parameters of the graph search that can stand in for stage 1 + stage 2a (g7_graph.cu).
struct GraphSearch {
    int32_t beam = 0, n_entries = 0, max_expansions = 0;
};

// Device status bits kept in the first word of a workspace.
enum : uint32_t { ST_OVERFLOW = 1u, ST_BAD_QUERY = 2u, ST_TIMEOUT = 4u, ST_BAD_INDEX = 8u };
constexpr int STATUS_WORD_CANARY = 8;   // status[8]: first damaged guard region found by the debug build's check

// ---------------------------------------------------------------------------------------------------------------
// Workspace layout (all offsets 256-byte aligned).
// ---------------------------------------------------------------------------------------------------------------
struct Params {
    int32_t B, nq, P, n_prune, k;
    int64_t maxc;                     // candidate capacity per query
};

// Whether a call cuts (on the device).  The load belongs beside a kernel's first ones, in front of the branch on it.
struct FirstCut {
    const int32_t *kept = nullptr;     // sampled candidates that would be kept; NULL: the call cuts
    int32_t most = 0;                  // with more of them it does not
#ifdef __CUDACC__
    __device__ __forceinline__ bool on() const { return kept == nullptr || __ldg(kept) <= most; }
#endif
};

constexpr int MAX_GUARDS = 64;
struct Layout {
    // debug builds (CHIMERA_DEBUG) put a 256-byte guard region behind every region below; guards[i] is its offset
    size_t guards[MAX_GUARDS];
    int n_guards;
    size_t status;        // uint32[64]
    size_t q_stage;       // float  [B, nq, D]        (host-entry staging of the queries)
    size_t out_ids;       // int32  [B, k]            (host-entry staging)
    size_t out_scores;    // float  [B, k]
    size_t qdig;          // int8   [3][table_rows(B*nq)][128], rows in table_row() order
    size_t qdig4;         // int8   [3][B*residual_rows(nq)][128]  the same for stage 4
    size_t table;         // int32  [B][K][nq]
    size_t table8;        // uint8  [B][K][coarse_pitch(nq)]  coarse copy: clamp(S >> 16, 0, 255), zeros past nq
    size_t part;          // uint64 [B][n_part][P][nq] partial top-P keys
    size_t probes;        // int32  [B][nq][P]
    size_t pq_gmax;       // int32  [B][pq_groups][nq] stages 1 + 2a together: largest score of each group of sample rows,
    size_t pq_thr;        // int32  [B*nq]            score bound per query-token row, padded to 32 rows,
    size_t pq_cnt;        // int32  [B*nq]            keys queued for the row,
    size_t pq_keys;       // uint64 [B*nq][pq_cap]    the keys,
    size_t pq_ovf;        // int32  [B]               1 = a queue of this query overflowed (redo by the table scan)
    size_t bitmap;        // uint32 [B][words], followed by the probe kernel's counters int32 [B][ceil(nq / 32)]
    size_t chunk_cnt;     // int32  [B][n_chunks]
    size_t cand;          // int32  [B][maxc]
    size_t n_cand;        // int32  [B]
    size_t ci;            // int32  [B][maxc]         exact CI of the contenders (of every candidate: generic q_len / tap)
    size_t lo;            // int32  [B][maxc]         lower bound on CI of every candidate
    size_t hi;            // int32  [B][maxc]         upper bound
    size_t cont;          // int32  [B][maxc]         contender ids, ascending
    size_t cand_rng;      // int2   [B][maxc]         (first token, length) of each candidate (bound scan)
    size_t cont_rng;      // int2   [B][maxc]         the same for the contenders
    size_t n_cont;        // int32  [B]
    size_t flt_theta;     // int32  [B][nq]           first cut (g3_filter.cu): thresholds,
    size_t flt_tab;       // uint8  [B][pitch]        one number per centroid (a batch at a time: rows of codes, g3_batch_scan.cu),
    size_t flt_over;      // that form's steps and listed centroids,
    size_t flt_mask;      // uint32 [B][ceil(K / 32)] centroids with a number above zero,
    size_t flt_hist;      // int32  [B][bins]         histogram of the bounds,
    size_t flt_parts;     // int32  histograms and counters of the threshold kernel's blocks (few queries)
    size_t flt_thr;       // int32  [B]               hi0 from which a candidate is a seed,
    size_t flt_slot;      // int32  [B][maxc]         place of each seed in the seed list,
    size_t flt_tau;       // int32  [B]               n_prune-th largest exact CI of the seeds (lower bound, without the cut),
    size_t flt_smp;       // int2   [CUT_SAMPLES]   CI and first bound of sampled candidates,
    size_t flt_vote;      // int32  [64]              how many of those would be kept, counters of the kernel that finds out,
    size_t flt_counts;    // int32  [B][slots]        kept candidates per slice
    size_t kept;          // int32  [B][maxc]         candidates that pass it, ascending
    size_t kept_rng;      // int2   [B][maxc]         their token ranges
    size_t n_kept;        // int32  [B]
    size_t n_seed;        // int32  [B]
    size_t n_rest;        // int32  [B]               kept candidates whose first upper bound does not decide
    size_t pruned;        // int32  [B][n_prune]
    size_t ranks;         // uint2  [B][words]        bitmap word, candidates before it (document -> candidate index);
                          //                          only with token lists, or where the first cut scans a batch at a time
    size_t partial_m;     // int32  [B][maxc][nq]     per (candidate, query token) best retrieved-token score, or the visit
                          //                          lists in its place (g3_visits.cuh); in the place of lo ... n_rest
    int64_t visit_nodes;  // nodes per query of those lists; 0 = the table
    size_t graph_vis;     // uint32 [B*nq][K/32]      visited centroids of the graph search (only with a centroid graph, and
                          //                          too many centroids for a bitmap in shared memory)
    size_t q_rot;         // float  [B, nq, D]        rotated queries (RaBitQ pipeline)
    size_t qdig_rot;      // int8   [3][B*residual_rows(nq)][128]  their digit planes for stage 4
    size_t n_pruned;      // int32  [B]
    size_t pruned_ci;     // int32  [B][n_prune] stage-3 score of each survivor (document-sharded search)
    size_t sel_scratch;   // int32  histograms and slice counts of the multi-block selection (few queries per call)
    size_t score4;        // float  [B][n_prune]
    size_t total;
    // derived sizes
    int32_t pq_stride;    // every pq_stride-th centroid tile is a sample tile; 0 = stages 1 and 2a run separately
    int32_t pq_cap;       // keys per queue
    int32_t pq_groups;    // groups of sample rows per query (one maximum each)
    int32_t n_part;       // partial lists per query in the probe stage
    int32_t probe_blocks; // blocks per query in the probe stage
    int64_t words;        // bitmap words per query
    int32_t n_chunks;     // bitmap chunks per query
};

constexpr int PROBE_WARPS = 8;          // warps per block in the probe stage (each keeps its own partial list)
constexpr int BITMAP_CHUNK_WORDS = 1024; // bitmap words per compaction block

Layout make_layout(const Index &ix, const Params &p);

// ---------------------------------------------------------------------------------------------------------------
// Error text (thread local) and helpers.
// ---------------------------------------------------------------------------------------------------------------
int fail(int code, const char *fmt, ...);
#define CHIMERA_CUDA(call)                                                                      \
    do {                                                                                        \
        cudaError_t e__ = (call);                                                               \
        if (e__ != cudaSuccess)                                                                 \
            return ::chimera::fail(CHIMERA_CUDA_ERROR, "%s: %s", #call, cudaGetErrorString(e__)); \
    } while (0)

// ---------------------------------------------------------------------------------------------------------------
// Profiling hooks (api.cu).
// ---------------------------------------------------------------------------------------------------------------
// Limit of the bounded device-side waits and the test hook that makes them run out (api.cu; chimera_test_wait_fault).
long long wait_limit_cycles();
int fault_skip_tma_loads();

enum Slot { SLOT_G1 = 0, SLOT_PROBE, SLOT_GATHER, SLOT_CI, SLOT_SELECT, SLOT_G4, SLOT_TOPK, SLOT_MISC, SLOT_CI_EXACT };
void count_launch(int slot, int n = 1);

// Dynamic shared memory above the default 48 KB.  The limit belongs to the kernel and not to a call, so every call sets the most that
// any call of the kernel takes: with its own size a search on another thread, of another index or other parameters, could lower
// the limit between this call's setting and its launch.
template <class... P>
cudaError_t allow_shared(void (*kernel)(P...), size_t most)
{
    return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)most);
}

// ---------------------------------------------------------------------------------------------------------------
// Launches of a search.  A search is a chain of up to two dozen short kernels on one stream, so the gaps between them are a
// good part of a small call.  Every kernel is launched as a programmatic dependent of the one before it: its blocks are
// placed as soon as that kernel's have exited, and pdl_entry(), the first thing every kernel does, waits until
// that kernel has finished and its writes are visible (one query against 10,000 documents: 142 -> 107 us).  EVERY kernel
// launched this way has to begin with pdl_entry(), on all its threads: the next kernel relies on this one to have waited.
// ---------------------------------------------------------------------------------------------------------------
template <class... P, class... A>
void launch(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, A &&...args)
{
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);       // (errors: cudaGetLastError() behind every launch)
}
#ifdef __CUDACC__
__device__ __forceinline__ void pdl_entry() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
// (No kernel lets its successor in earlier, with griddepcontrol.launch_dependents: blocks that wait hold shared memory, and
// with it L1, of the kernel they wait for.  Measured with the trigger behind pdl_entry(), in all kernels: Mid, batch 256, 9.2
// -> 12.1 ms; in the short ones only: 9.2 -> 9.6 ms, one query 184 -> 214 us.)
#endif

// ---------------------------------------------------------------------------------------------------------------
// Stage launchers (one per .cu file).  Each only enqueues kernels on `st` and returns a chimera_status.
// ---------------------------------------------------------------------------------------------------------------
int build_index_device(Index &ix, const float *centroids, const int32_t *doclens, cudaStream_t st);
// rows x D float32 in [-1, 1] -> three int8 digit planes [3][rows][128] (zero padded, dimensions in digit_dim() order);
// out-of-range elements set ST_BAD_QUERY.  tiles: planes of table_rows(rows) rows in table_row() order, the padding not written.
// dig4 (may be NULL): the same planes for stage 4, rows = query tokens (q_len of them per query) in score_row() order,
// padded to residual_rows(q_len) per query; the padding is not written.  dig may be NULL then.
// clear / clear_n (may be NULL / 0): 32-bit words set to zero on the side, for a later kernel of the same call.
int launch_digits(const float *x, int64_t rows, int D, int nbits, int8_t *dig, bool tiles, int8_t *dig4, int q_len,
                  uint32_t *status, cudaStream_t st, uint32_t *clear = nullptr, int64_t clear_n = 0);

// table8 may be NULL (no coarse copy wanted).
int launch_score_table(const Index &ix, const Params &p, const float *queries, int8_t *qdig, int8_t *qdig4, int32_t *table,
                       uint8_t *table8, uint32_t *status, cudaStream_t st, uint32_t *clear = nullptr, int64_t clear_n = 0);
// done (may be NULL): counters int32 [B][ceil(nq / 32)], zero before; the probe kernel's last block then folds its lists
// itself instead of a second kernel.
int launch_probes(const Index &ix, const Params &p, const Layout &L, const int32_t *table, unsigned long long *part,
                  int32_t *probes, int32_t *done, cudaStream_t st);
// Stages 1 and 2a together (g1_score_table.cu), used when the layout has pq_stride > 0, and its probe-side pieces
// (g2_probe.cu): the sample's top nprobe and bounds; the final top nprobe from sample list and queues, with the table
// scan as the fallback for queries whose queue overflowed.  keep_table: the table is wanted beside the probes; without it
// only the sample's tiles are written, and launch_probe_merge (given the query digits) has the rest made for those queries.
int probe_sample_stride(int64_t K, int nq, int P);       // host arithmetic only
int probe_queue_stride(const Index &ix, const Params &p);
int probe_queue_cap();
int probe_sample_groups(const Index &ix, int stride);
int launch_score_table_probes(const Index &ix, const Params &p, const Layout &L, const float *queries, int8_t *qdig,
                              int8_t *qdig4,
                              int32_t *table, bool keep_table, uint8_t *table8, char *ws, uint32_t *status, cudaStream_t st,
                              uint32_t *clear = nullptr, int64_t clear_n = 0);
int launch_score_table_redo(const Index &ix, const Params &p, const Layout &L, const int8_t *qdig, int32_t *table,
                            const int32_t *redo, uint32_t *status, cudaStream_t st);
int launch_probe_sample(const Index &ix, const Params &p, const Layout &L, const int32_t *table, char *ws,
                        int n_sample_tiles, cudaStream_t st);
int launch_probe_merge(const Index &ix, const Params &p, const Layout &L, int32_t *table, const int8_t *redo_qdig, char *ws,
                       uint32_t *status, cudaStream_t st);
// bitmap_clear: the bitmap is zero already.  ranks, rng (the candidates' token ranges), cont_scratch (rows of which the
// contender step's histogram is cleared): each may be NULL.
int launch_gather(const Index &ix, const Params &p, const Layout &L, const int32_t *probes, uint32_t *bitmap,
                  bool bitmap_clear, int32_t *chunk_cnt, int32_t *cand, int32_t *n_cand, uint2 *ranks, int2 *rng,
                  int32_t *cont_scratch, uint32_t *status, cudaStream_t st);
bool contenders_split(const Index &ix, const Params &p);
int contender_hist_entries();
// Token-level posting lists for the refinements, unless they are there, and copies of `n` arrays ([T][words] 32-bit words each,
// document-major) in their order, so that a list's codes are one contiguous run instead of a scattered sector each
// (index_build.cu).  The copies are complete when the call returns.  Every dst is NULL, with CHIMERA_OK, when they would take
// more than a quarter of the free memory (the kernels then gather through the token ids), and on every error.
struct ListOrderCopy {
    const void *src;
    int words;
    void *dst;
};
int build_lists_and_copies(Index &ix, ListOrderCopy *copies, int n, ListMemory &mem, cudaStream_t st);
// Candidate refinement with partial scores (Algorithm 2): fprime[b][j] for every candidate.
int64_t visit_list_nodes(const Index &ix, const Params &p);
int launch_partial_scores(const Index &ix, const Params &p, const Layout &L, const int8_t *qdig,
                          const int32_t *table, const int32_t *probes, const uint2 *ranks, const int32_t *n_cand,
                          void *partial_m, int32_t *fprime, cudaStream_t st);
int launch_filter_contenders(const Index &ix, const Params &p, const Layout &L, const int32_t *kept, const int2 *kept_rng,
                             const int32_t *n_kept, const int32_t *lo, const int32_t *hi, int32_t *cont, int2 *cont_rng,
                             int32_t *n_cont, char *ws, cudaStream_t st);
bool coarse_supported(int nq);
int coarse_pitch(int nq);       // bytes of an 8-bit row
int launch_coarse_table(const Index &ix, const Params &p, const int32_t *table, uint8_t *table8, cudaStream_t st);
// The candidates' token ranges (corpora with fewer than 2^31 tokens); also clears the contender step's histograms at the
// head of its scratch rows (int32 [B][maxc]) where launch_contenders will use them.
int launch_cand_ranges(const Index &ix, const Params &p, const int32_t *cand, const int32_t *n_cand, int2 *rng,
                       int32_t *cont_scratch, cudaStream_t st);
// rng: those ranges (may be NULL: per-document offset lookups instead).  cut (may be NULL, else with ranges): a call that cuts
// does nothing here.
int launch_coarse_bounds(const Index &ix, const Params &p, const uint8_t *table8, const int32_t *cand,
                         const int32_t *n_cand, int32_t *lo, int32_t *hi, const int2 *rng, const FirstCut *cut, cudaStream_t st);
// Upper bounds of what a call that cuts has kept.  mask: [B][ceil(K / 32)] bits of the centroids near a query token, or NULL;
// theta, tau: the cut's.  rng: token ranges; (CI, 0) stands for a document whose exact CI is known.  rest: int32 [B][maxc] scratch,
// n_rest: int32 [B], zero before.
int launch_kept_bounds(const Index &ix, const Params &p, const uint8_t *table8, const uint32_t *mask, const int32_t *theta,
                       const int32_t *tau, const int2 *rng, const int32_t *n_docs, int32_t *hi, int32_t *rest, int32_t *n_rest,
                       const FirstCut &cut, cudaStream_t st);
// First cut of the candidates by an upper bound from one number per token (g3_filter.cu).  launch_filter_scan leaves the
// bounds in hi0 and the best ~2 n_prune candidates in seed / seed_rng (their number in the workspace's n_seed);
// launch_filter_keep takes the seeds' exact CI and writes the candidates that can still be in the top n_prune, ascending;
// launch_filter_contenders narrows them down by the 8-bit upper bounds.  Where a sample shows that the cut would keep most
// candidates, there are no seeds, all candidates are kept, and the contenders are found by the 8-bit lower bounds.
constexpr int CUT_QUERIES = 16, CUT_SAMPLES = 4096;
FirstCut first_cut(const Params &p, const Layout &L, char *ws);
bool filter_used(const Index &ix, const Params &p);
bool filter_mask_used(const Index &ix, const Params &p, bool batch);      // the masks are written
bool batch_scan_used(const Index &ix, const Params &p);       // ... and scans for all queries at once (g3_batch_scan.cu)
int batch_group(const Params &p);                             // that many side by side
size_t batch_table_bytes(const Index &ix, const Params &p);
// ... with the numbers of listed centroids, int32 [B], at its end.
size_t batch_over_bytes(const Params &p);
size_t filter_table_pitch(const Index &ix);
int filter_hist_bins();
int filter_count_slots();
size_t filter_parts_bytes(const Index &ix, const Params &p);
// batch: by the batch's form, which needs the workspace's ranks.
int launch_filter_scan(const Index &ix, const Params &p, const Layout &L, bool batch, const int32_t *table, uint8_t *table8,
                       const int32_t *cand, const int32_t *n_cand, int32_t *hi0, int32_t *seed,
                       int2 *seed_rng, char *ws, cudaStream_t st);
int launch_filter_keep(const Index &ix, const Params &p, const Layout &L, const int32_t *cand,
                       const int32_t *n_cand, const int32_t *hi0, const int32_t *seed_ci, int32_t *kept,
                       int2 *kept_rng, int32_t *n_kept, char *ws, cudaStream_t st);
// scratch: an int32 [B][maxc] array that is free during this step.
// rng / cont_rng (may be NULL): the candidates' token ranges and where to put those of the contenders.
int launch_contenders(const Index &ix, const Params &p, const int32_t *cand, const int32_t *n_cand, const int32_t *lo,
                      const int32_t *hi, int32_t *cont, int32_t *n_cont, int32_t *scratch, const int2 *rng,
                      int2 *cont_rng, cudaStream_t st);
// rng (may be NULL, used when blocks_cap > 0): the token ranges of the listed documents, in list order; (CI, 0) stands
// for a document whose CI is known.
int launch_centroid_interaction(const Index &ix, const Params &p, const int32_t *table, const int32_t *cand,
                                const int32_t *n_cand, int32_t *ci, int blocks_cap, int slot, const int2 *rng,
                                cudaStream_t st);
// pruned_ci (may be NULL): the score of each kept document, INT_MIN in the padding.
// scratch: select_split_scratch_bytes() bytes (few queries per call: several blocks per query), or NULL.
enum { GATHER_L2, GATHER_SHARED, GATHER_RANGES };                 // where the bits of a query's candidates are set
int gather_form(const Index &ix, const Params &p);
double expected_candidates(const Index &ix, const Params &p);     // of a query
bool select_few_used(const Index &ix, const Params &p);           // a selection among all candidates is prepared for few of many
bool select_split_used(const Index &ix, const Params &p);
size_t select_split_scratch_bytes(const Index &ix, const Params &p);
int launch_select(const Index &ix, const Params &p, const int32_t *cand, const int32_t *n_cand, const int32_t *ci,
                  int32_t *pruned, int32_t *n_pruned, int32_t *pruned_ci, int32_t *scratch, bool many, cudaStream_t st);
// Document-sharded search: the global top-n_prune of the shards' lists and the final top-k merge.
int launch_shard_export(const Params &p, const int32_t *pruned, const int32_t *pruned_ci, int64_t doc_base,
                        int32_t *out_ids, int32_t *out_ci, cudaStream_t st);
int launch_shard_select(const Params &p, const int32_t *all_ids, const int32_t *all_ci, int world, int64_t doc_base,
                        int64_t n_local, int32_t *pruned, int32_t *n_pruned, cudaStream_t st);
int launch_add_base(int32_t *ids, int64_t n, int64_t doc_base, cudaStream_t st);
int launch_shard_merge_topk(const int32_t *all_ids, const float *all_scores, int world, int B, int k, int32_t *out_ids,
                            float *out_scores, cudaStream_t st);
// qdig4 = the query digit planes in stage 4's own row order.
int launch_residual_scores_umma(const Index &ix, const Params &p, const float *queries, const int8_t *qdig,
                                const int32_t *table, const int32_t *pruned, float *score4, uint32_t *status,
                                cudaStream_t st);
int launch_rabitq_scores_umma(const Index &ix, const Params &p, const float *q_rot, const int8_t *qdig_rot,
                              const int32_t *pruned, float *score4, uint32_t *status, cudaStream_t st);
// g7_graph.cu
int build_graph(Index &ix, const float *centroids, int degree, cudaStream_t st);
size_t graph_scratch_bytes(const Index &ix, int64_t n_tokens);
size_t graph_workspace_bytes(const Index &ix, int64_t n_tokens);     // of a search that does not want the visited sets
int graph_search_warps(const Index &ix, int64_t n_tokens);           // warps of a search's block: 2 or 4
int check_graph_params(const Index &ix, const GraphSearch &g, int nprobe);
// visited: graph_scratch_bytes(ix, n_tokens) bytes of scratch, holding the visited sets afterwards if want_visited;
// graph_workspace_bytes(ix, n_tokens) otherwise;
// out_scores / out_nvis may be NULL.
int launch_graph_probes(const Index &ix, const float *queries, int64_t n_tokens, int nprobe, const GraphSearch &g,
                        uint32_t *visited, bool want_visited, int32_t *out_probes, int32_t *out_scores, int32_t *out_nvis,
                        cudaStream_t st);
// rabitq.cu
int transpose_rotation(const Index &ix, const float *rotation, float **rot_t, cudaStream_t st);   // (allocates)
int launch_rotate(const Index &ix, const Params &p, const float *queries, float *q_rot, cudaStream_t st);
int launch_rabitq_partial(const Index &ix, const Params &p, const Layout &L, const int8_t *qdig_rot,
                          const int32_t *probes, const uint2 *ranks, const int32_t *n_cand, void *partial_m,
                          int32_t *fprime_bits, cudaStream_t st);
int launch_topk(const Index &ix, const Params &p, const int32_t *pruned, const float *score4, int32_t *out_ids,
                float *out_scores, cudaStream_t st);

// ---------------------------------------------------------------------------------------------------------------
// Debug build (-DCHIMERA_DEBUG, libchimera_debug.so): every index that a kernel is about to gather through (centroid
// id, document id, token position, candidate rank) is checked first.  An index out of range sets ST_BAD_INDEX in the
// status word of the running search and is replaced by 0 (DBG_*) or its access is skipped (DBG_*_OK), so the kernel
// never touches memory outside its arrays.  The limits and the status pointer of the running search live in one
// device variable, so a debug build serves one search at a time.  In release builds the macros vanish.
// ---------------------------------------------------------------------------------------------------------------
#ifdef CHIMERA_DEBUG
struct DbgLimits { uint32_t *status; long long K, N, T, maxc; };
extern __device__ DbgLimits chimera_dbg;
__device__ __forceinline__ bool dbg_in_range(long long x, long long n)
{
    if (x >= 0 && x < n) return true;
    if (chimera_dbg.status) atomicOr(chimera_dbg.status, ST_BAD_INDEX);
    return false;
}
template <class I> __device__ __forceinline__ I dbg_index(I x, long long n) { return dbg_in_range((long long)x, n) ? x : (I)0; }
#define DBG_CID(c) ::chimera::dbg_index((c), ::chimera::chimera_dbg.K)
#define DBG_DOC(d) ::chimera::dbg_index((d), ::chimera::chimera_dbg.N)
#define DBG_TOK(t) ::chimera::dbg_index((t), ::chimera::chimera_dbg.T)
#define DBG_DOC_OK(d) ::chimera::dbg_in_range((long long)(d), ::chimera::chimera_dbg.N)
#define DBG_RANK_OK(r) ::chimera::dbg_in_range((long long)(r), ::chimera::chimera_dbg.maxc)
#else
#define DBG_CID(c) (c)
#define DBG_DOC(d) (d)
#define DBG_TOK(t) (t)
#define DBG_DOC_OK(d) true
#define DBG_RANK_OK(r) true
#endif
// Host side (api.cu): publish the running search's limits / fill and check the guard regions (no-ops in release builds).
int debug_begin_search(const Index &ix, const Params &p, const Layout &L, void *workspace, cudaStream_t st);

// Order of the dimensions in a digit row: position -> dimension.  A contraction does not care as long as both operands
// agree, so the order is the one in which packed codes expand with one shift and one mask per four dimensions (stage 4):
// (word >> 2 j) & 0x03030303 holds dimensions j, 4 + j, 8 + j, 12 + j of the word's 16 2-bit codes, and
// (word >> j) & 0x01010101 dimensions j, 8 + j, 16 + j, 24 + j of its 32 1-bit codes.
__host__ __device__ __forceinline__ int digit_dim(int pos, int nbits)
{
    return nbits == 2 ? (pos & ~15) | (pos & 3) << 2 | (pos >> 2 & 3) : (pos & ~31) | (pos & 3) << 3 | (pos >> 2 & 7);
}

// Stage 1 on the tensor cores: rows of the query digit planes (whole tiles of 32), and the row of query token i of a batch.
// Within a tile, tokens 8 g ... 8 g + 7 sit in rows 2 g, 2 g + 1, 8 + 2 g, 8 + 2 g + 1, ...: the accumulator columns that the
// same thread reads back, so that it stores eight neighbouring scores of a centroid and four threads a whole row of 32.
__host__ __device__ __forceinline__ int64_t table_rows(int64_t rows) { return (rows + 31) & ~(int64_t)31; }
__host__ __device__ __forceinline__ int64_t table_row(int64_t i) { return (i & ~(int64_t)31) | (i << 2 & 24) | (i >> 2 & 6) | (i & 1); }

// Stage 4 on the tensor cores: rows per query of its digit planes, and the row of query token i.  Within 16 tokens, tokens
// 4 g ... 4 g + 3 sit in rows 2 g, 2 g + 1, 8 + 2 g, 8 + 2 g + 1: the accumulator columns that the same thread reads back,
// so that its four score-table entries are one 16-byte load.
__host__ __device__ __forceinline__ int residual_rows(int q_len) { return q_len <= 32 ? 32 : q_len <= 64 ? 64 : 128; }
__host__ __device__ __forceinline__ int score_row(int i) { return (i & ~15) | (i & 2) << 2 | (i >> 1 & 6) | (i & 1); }

// ---------------------------------------------------------------------------------------------------------------
// Device helpers.
// ---------------------------------------------------------------------------------------------------------------
__device__ __forceinline__ int warp_sum(int v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}
// (first token, length) of a document (corpora with fewer than 2^31 tokens).
__device__ __forceinline__ int2 doc_range(const int64_t *doc_off, int32_t d)
{
    d = DBG_DOC(d);
    const int64_t t0 = __ldg(doc_off + d);
    return make_int2((int)t0, (int)(__ldg(doc_off + d + 1) - t0));
}
__device__ __forceinline__ float warp_sum(float v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}
__device__ __forceinline__ unsigned long long warp_max(unsigned long long v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        unsigned long long w = __shfl_xor_sync(0xffffffffu, v, o);
        v = w > v ? w : v;
    }
    return v;
}

// Order-preserving key of (score desc, id asc): a larger key is a better entry.
__device__ __forceinline__ unsigned long long key_int(int32_t score, int32_t id)
{
    return ((unsigned long long)((uint32_t)score ^ 0x80000000u) << 32) | (uint32_t)(0xFFFFFFFFu - (uint32_t)id);
}
__device__ __forceinline__ int32_t key_id(unsigned long long key) { return (int32_t)(0xFFFFFFFFu - (uint32_t)key); }

}  // namespace chimera
