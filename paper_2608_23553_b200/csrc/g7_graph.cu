// Proximity graph over the centroids and its search: the replacement of the exhaustive centroid scan (stage 1 +
// stage 2a) that the paper uses (Sec. 3.1: a proximity-graph index built on the IVF centroids; Algorithm 1, line
// searchCAGRA; Sec. 2.3 for how such a graph is searched).
//
// Graph (index time): node c is linked to the `degree` other centroids with the largest fixed-point inner product
// S_fx(c, c'), ties towards the smaller id, best first.  It is built with the library's own exact machinery: the
// centroids take the place of query tokens in the stage-1 tensor-core kernel and stage 2a picks each row's best
// degree + 1 entries, of which the centroid itself is dropped.
//
// Search (query time): a block of two or four warps per query token runs a best-first search with a bounded result list:
//   - the entry points floor(j K / n_entries), j < n_entries, are visited (scored, marked, offered to the list);
//   - repeatedly the first list member that has not been expanded is expanded: each of its graph neighbours that was
//     never visited is visited; the search ends when every list member is expanded or after max_expansions expansions;
//   - the list keeps the best `beam` visited centroids by (score descending, id ascending).
// The score is the exact S_fx(q, c) = floor((sum_d Xq[d] Xc[d] + 2^19) / 2^20) in 64-bit integers, so the list after
// each step is the best `beam` of everything offered so far whatever the order of evaluation, and the visited set, the
// probes and their scores are reproducible bit for bit.  The list lives in the first warp's registers (two 64-bit keys per
// lane, sorted by slot = lane + 32 j), the visited set is a bitmap in shared memory (in global memory above 2^20 centroids).
#include "common.cuh"

namespace chimera {

// Xc[c][d] = rint(centroid * 2^22), recombined from the three balanced base-256 digit planes of the index.
__global__ void xc_kernel(const int8_t *__restrict__ cdig, int64_t K, int D, int nbits, int32_t *__restrict__ xc)
{
    const int64_t n = K * D;
    const int64_t plane = K * 128;
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x) {
        const int64_t c = e / D;
        const int i = (int)(e % D);                          // (D is a multiple of 32: positions below D hold all dimensions)
        const int64_t at = c * 128 + i;
        xc[c * D + digit_dim(i, nbits)] = (int)cdig[at] + 256 * (int)cdig[plane + at] + 65536 * (int)cdig[2 * plane + at];
    }
}

// probes [rows][R + 1] of centroids c0 .. c0 + rows - 1 (each row best first) -> graph rows: the centroid itself is
// dropped (or the last entry, when identical twins with smaller ids pushed it out of the list).
__global__ void graph_rows_kernel(const int32_t *__restrict__ probes, int64_t c0, int rows, int R,
                                  int32_t *__restrict__ graph)
{
    const int r = blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= rows) return;
    const int32_t *pr = probes + (int64_t)r * (R + 1);
    int32_t *out = graph + (c0 + r) * R;
    int w = 0;
    for (int e = 0; e <= R && w < R; ++e)
        if (pr[e] != (int32_t)(c0 + r)) out[w++] = pr[e];
}

int build_graph(Index &ix, const float *centroids, int R, cudaStream_t st)
{
    if (R < 1 || R > CHIMERA_MAX_NPROBE - 1 || R > ix.K - 1)
        return fail(CHIMERA_INVALID_ARG, "degree must be in [1, min(%d, n_centroids - 1)], got %d", CHIMERA_MAX_NPROBE - 1, R);
    cudaFree(ix.graph);
    cudaFree(ix.xc);
    ix.graph = nullptr;
    ix.xc = nullptr;
    ix.graph_deg = 0;
    int32_t *graph = nullptr, *xc = nullptr;
    char *ws = nullptr;
    float *qbuf = nullptr;
    auto cleanup = [&]() { cudaFree(ws); cudaFree(qbuf); };
    auto drop = [&]() { cleanup(); cudaFree(graph); cudaFree(xc); };
    // pseudo-queries of 32 centroids each; as many per call as keep the score table near 512 MB
    constexpr int NQ = 32;
    int64_t bq = (512LL << 20) / (ix.K * NQ * 4);
    if (bq < 1) bq = 1;
    if (bq > 64) bq = 64;
    const int64_t need = (ix.K + NQ - 1) / NQ;
    if (bq > need) bq = need;
    Params p;
    p.B = (int32_t)bq; p.nq = NQ; p.P = R + 1; p.n_prune = 1; p.k = 1; p.maxc = 1;
    const Layout L = make_layout(ix, p);
    const int rows_per_call = (int)bq * NQ;
    cudaError_t e = cudaMalloc(&graph, sizeof(int32_t) * (size_t)ix.K * R);
    if (e == cudaSuccess) e = cudaMalloc(&xc, sizeof(int32_t) * (size_t)ix.K * ix.D);
    if (e == cudaSuccess) e = cudaMalloc(&ws, L.total);
    if (e == cudaSuccess) e = cudaMalloc(&qbuf, sizeof(float) * (size_t)rows_per_call * ix.D);
    if (e != cudaSuccess) {
        drop();
        return fail(CHIMERA_CUDA_ERROR, "cudaMalloc (centroid graph): %s", cudaGetErrorString(e));
    }
    xc_kernel<<<(unsigned)(8 * ix.sm_count), 256, 0, st>>>(ix.cdig, ix.K, ix.D, ix.nbits, xc);
    uint32_t *status = (uint32_t *)(ws + L.status);
    int8_t *qdig = (int8_t *)(ws + L.qdig);
    int32_t *table = (int32_t *)(ws + L.table);
    unsigned long long *part = (unsigned long long *)(ws + L.part);
    int32_t *probes = (int32_t *)(ws + L.probes);
    int rc = CHIMERA_OK;
    for (int64_t c0 = 0; c0 < ix.K && rc == CHIMERA_OK; c0 += rows_per_call) {
        const int rows = (int)(ix.K - c0 < rows_per_call ? ix.K - c0 : rows_per_call);
        e = cudaMemcpyAsync(qbuf, centroids + c0 * ix.D, sizeof(float) * (size_t)rows * ix.D, cudaMemcpyDeviceToDevice, st);
        if (e == cudaSuccess && rows < rows_per_call)
            e = cudaMemsetAsync(qbuf + (size_t)rows * ix.D, 0, sizeof(float) * (size_t)(rows_per_call - rows) * ix.D, st);
        if (e != cudaSuccess) { rc = fail(CHIMERA_CUDA_ERROR, "copy (centroid graph): %s", cudaGetErrorString(e)); break; }
        if ((rc = launch_score_table(ix, p, qbuf, qdig, nullptr, table, nullptr, status, st))) break;
        if ((rc = launch_probes(ix, p, L, table, part, probes, nullptr, st))) break;
        graph_rows_kernel<<<(unsigned)((rows + 127) / 128), 128, 0, st>>>(probes, c0, rows, R, graph);
    }
    if (rc == CHIMERA_OK) {
        e = cudaGetLastError();
        if (e == cudaSuccess) e = cudaStreamSynchronize(st);
        if (e != cudaSuccess) rc = fail(CHIMERA_CUDA_ERROR, "centroid graph build: %s", cudaGetErrorString(e));
    }
    if (rc != CHIMERA_OK) {
        cudaStreamSynchronize(st);
        drop();
        return rc;
    }
    cleanup();
    ix.graph = graph;
    ix.xc = xc;
    ix.graph_deg = R;
    return CHIMERA_OK;
}

// ------------------------------------------------------------------------------------------------ search ---------
// List key: a larger key ranks first.  Score in the high word, then the id (smaller id = larger key), and in bit 0
// whether the member is still to be expanded; ids differ by at least 2 in this field, so the flag never decides an
// order.  A valid key is non-zero.
__device__ __forceinline__ unsigned long long gp_key(int32_t score, int32_t id)
{
    return ((unsigned long long)((uint32_t)score ^ 0x80000000u) << 32) | ((uint32_t)(0x7FFFFFFF - id) << 1) | 1ull;
}
__device__ __forceinline__ int32_t gp_id(unsigned long long key) { return 0x7FFFFFFF - (int32_t)((uint32_t)key >> 1); }
__device__ __forceinline__ int32_t gp_score(unsigned long long key) { return (int32_t)((uint32_t)(key >> 32) ^ 0x80000000u); }

// grid (tokens), one block of WARPS warps per query token.  The search is a chain -- best unexpanded member -> its neighbours ->
// which are new -> their rows -> their scores -> the list -- so it is latency that counts: the visited set is a bitmap in
// shared memory (SHARED; written out at the end when wanted), all warps fetch and score the new centroids of a step
// together, and warp 0 keeps the list in registers and looks only at scores that rank inside it.  Many tokens hide that chain,
// and then the instructions count: eight lanes score a centroid (a warp per centroid, its sum by two hardware reductions, took 94
// instructions each over all warps), a row's address is one 32 x 32-bit multiply-add, places in s_ids come from votes, keys
// are compared as they are, and only lists of more than 32 members (WIDE) have a second key per lane.
// Mid, beam 32, 256 entries: 2,048 tokens 470 -> 244 us with two warps (all blocks resident at once; four: 268), 32 tokens 192 -> 116
// with four (two: 155), 8,192 tokens 1,492 -> 718.  Two rows in flight per eight lanes: 300.  (Which of the two: graph_search_warps.)
// visited (NULL: not wanted; !SHARED: [tokens][vwords] zeroed by the caller).
template <bool SHARED, bool WIDE, int WARPS>
__global__ void __launch_bounds__(WARPS * 32, 32 / WARPS)
graph_probe_kernel(const float *__restrict__ queries, int D, const int32_t *__restrict__ xc,
                   const int32_t *__restrict__ graph, int R, int64_t K, int n_entries, int beam, int max_exp,
                   int nprobe, uint32_t *__restrict__ visited, int64_t vwords, int32_t *__restrict__ out_probes,
                   int32_t *__restrict__ out_scores, int32_t *__restrict__ out_nvis)
{
    pdl_entry();
    constexpr int BATCH = WARPS * 32;                    // centroids of a step, at most
    extern __shared__ uint32_t s_vis[];
    __shared__ int32_t s_ids[BATCH], s_sc[BATCH];
    __shared__ int s_n, s_next;                          // centroids of the step; the member to expand (-1: none)
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int64_t token = blockIdx.x;
    // eight lanes score a centroid: lane l8 has dimensions 32 q + 4 l8 ... + 3 of it, q < D / 32
    const int l8 = lane & 7, quads = D >> 5;
    int xq[4][4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const float4 v = q < quads ? __ldg(reinterpret_cast<const float4 *>(queries + token * D) + 8 * q + l8) : make_float4(0.f, 0.f, 0.f, 0.f);
        xq[q][0] = __float2int_rn(fminf(fmaxf(v.x, -1.0f), 1.0f) * 4194304.0f);
        xq[q][1] = __float2int_rn(fminf(fmaxf(v.y, -1.0f), 1.0f) * 4194304.0f);
        xq[q][2] = __float2int_rn(fminf(fmaxf(v.z, -1.0f), 1.0f) * 4194304.0f);
        xq[q][3] = __float2int_rn(fminf(fmaxf(v.w, -1.0f), 1.0f) * 4194304.0f);
    }
    uint32_t *vis = SHARED ? s_vis : visited + token * vwords;
    if (SHARED)
        for (int w = tid; w < (int)vwords; w += BATCH) s_vis[w] = 0u;
    if (tid == 0) s_n = 0;
    __syncthreads();

    const char *const xc_lane = reinterpret_cast<const char *>(xc) + 16 * l8;
    const uint32_t row_bytes = 4u * (uint32_t)D;
    unsigned long long key0 = 0ull, key1 = 0ull;         // warp 0: list slots lane and (WIDE) 32 + lane, best first
    int n_vis = 0;

    // offer a scored centroid (warp-uniform argument) to the list
    auto offer = [&](unsigned long long x) {
        // (x is no member: where the flags differ the ids do)
        int pos = __popc(__ballot_sync(0xffffffffu, key0 > x));
        if (WIDE) pos += __popc(__ballot_sync(0xffffffffu, key1 > x));
        if (pos >= beam) return;                          // ranks behind a full list
        const unsigned long long up0 = __shfl_up_sync(0xffffffffu, key0, 1);
        if (WIDE) {
            const unsigned long long up1 = __shfl_up_sync(0xffffffffu, key1, 1);
            const unsigned long long last0 = __shfl_sync(0xffffffffu, key0, 31);
            const int s1 = 32 + lane;
            if (s1 > pos) key1 = lane == 0 ? last0 : up1;
            else if (s1 == pos) key1 = x;
            if (s1 >= beam) key1 = 0ull;
        }
        if (lane > pos) key0 = up0;
        else if (lane == pos) key0 = x;
        if (lane >= beam) key0 = 0ull;                    // the member pushed past the end falls off
    };
    // this thread's centroid of the step (-1: none; whole warps): into s_ids when it was never visited (order does not matter:
    // the list is the best `beam` of everything offered)
    auto collect = [&](int32_t n) {
        bool fresh = false;
        if (n >= 0) {
            n = DBG_CID(n);
            const uint32_t bit = 1u << (n & 31);
            fresh = (atomicOr(&vis[n >> 5], bit) & bit) == 0u;
        }
        const unsigned who = __ballot_sync(0xffffffffu, fresh);
        if (who == 0u) return;
        int at = 0;
        if (lane == 0) at = atomicAdd(&s_n, __popc(who));
        at = __shfl_sync(0xffffffffu, at, 0);
        if (fresh) s_ids[at + __popc(who & ((1u << lane) - 1u))] = n;
    };
    // the step's centroids (at most BATCH): scored by all warps, offered by warp 0.  Two barriers; s_n is 0 afterwards.
    auto score_and_offer = [&]() {
        __syncthreads();
        const int cnt = s_n;
        for (int k0 = 4 * warp; k0 < cnt; k0 += 4 * WARPS) {
            const int k = k0 + (lane >> 3);                  // (past the end: the last one again)
            const char *row = xc_lane + (uint64_t)(uint32_t)s_ids[k < cnt ? k : cnt - 1] * row_bytes;
            int4 v[4];
#pragma unroll
            for (int q = 0; q < 4; ++q)
                if (q < quads) v[q] = __ldg(reinterpret_cast<const int4 *>(row + 128 * q));
            // exact S_fx(q, c): |s| < 2^46
            long long s = 0;
#pragma unroll
            for (int q = 0; q < 4; ++q)
                if (q < quads)
                    s += (long long)xq[q][0] * v[q].x + (long long)xq[q][1] * v[q].y + (long long)xq[q][2] * v[q].z +
                         (long long)xq[q][3] * v[q].w;
#pragma unroll
            for (int o = 4; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
            if (l8 == 0 && k < cnt) s_sc[k] = (int32_t)((s + (1LL << 19)) >> 20);
        }
        __syncthreads();
        if (warp == 0) {
            n_vis += cnt;
            for (int k0 = 0; k0 < cnt; k0 += 32) {
                const int k = k0 + lane;
                const unsigned long long mine = k < cnt ? gp_key(s_sc[k], s_ids[k]) : 0ull;
                for (uint32_t left = __ballot_sync(0xffffffffu, k < cnt); left;) {
                    // the keys that rank inside the list as it is now (it only gets better)
                    const unsigned long long last = WIDE && beam > 32 ? __shfl_sync(0xffffffffu, key1, beam - 33)
                                                                     : __shfl_sync(0xffffffffu, key0, beam - 1);
                    left &= __ballot_sync(0xffffffffu, mine > last);
                    if (!left) break;
                    const int src = __ffs(left) - 1;
                    left &= left - 1;
                    offer(__shfl_sync(0xffffffffu, mine, src));
                }
            }
            if (lane == 0) s_n = 0;
        }
    };

    for (int j0 = 0; j0 < n_entries; j0 += BATCH) {
        const int j = j0 + tid;
        collect(j < n_entries ? (int32_t)(((long long)j * K) / n_entries) : -1);
        score_and_offer();
        __syncthreads();
    }
    for (int done = 0; done < max_exp; ++done) {
        if (warp == 0) {
            const uint32_t u0 = __ballot_sync(0xffffffffu, (key0 & 1ull) != 0ull);
            const uint32_t u1 = WIDE ? __ballot_sync(0xffffffffu, (key1 & 1ull) != 0ull) : 0u;
            int32_t p = -1;                              // every member expanded
            if (u0) {
                const int src = __ffs(u0) - 1;
                p = gp_id(__shfl_sync(0xffffffffu, key0, src));
                if (lane == src) key0 &= ~1ull;
            } else if (u1) {
                const int src = __ffs(u1) - 1;
                p = gp_id(__shfl_sync(0xffffffffu, key1, src));
                if (lane == src) key1 &= ~1ull;
            }
            if (lane == 0) s_next = p;
        }
        __syncthreads();
        const int32_t p = s_next;
        if (p < 0) break;
        if (warp * 32 < R) collect(tid < R ? __ldg(graph + (int64_t)p * R + tid) : -1);          // (R <= 63)
        score_and_offer();
    }
    if (warp == 0) {
        for (int r = lane; r < nprobe; r += 32) {
            const unsigned long long k = r < 32 ? key0 : key1;   // r = lane or lane + 32
            out_probes[token * nprobe + r] = k ? gp_id(k) : -1;
            if (out_scores) out_scores[token * nprobe + r] = k ? gp_score(k) : INT32_MIN;
        }
        if (out_nvis && lane == 0) out_nvis[token] = n_vis;
    }
    if (SHARED && visited)
        for (int w = tid; w < (int)vwords; w += BATCH) visited[token * vwords + w] = s_vis[w];
}

size_t graph_scratch_bytes(const Index &ix, int64_t n_tokens)
{
    return (size_t)n_tokens * (size_t)((ix.K + 31) / 32) * sizeof(uint32_t);
}

// The search keeps the visited set in shared memory up to a million centroids.
constexpr size_t VISITED_SMEM = 128 * 1024;
static bool visited_in_shared(const Index &ix) { return (size_t)((ix.K + 31) / 32) * sizeof(uint32_t) <= VISITED_SMEM; }
size_t graph_workspace_bytes(const Index &ix, int64_t n_tokens)
{
    return visited_in_shared(ix) ? 0 : graph_scratch_bytes(ix, n_tokens);
}

// Warps per token: two where they make the search end in fewer rounds of resident blocks.  Registers hold 8 blocks of four warps or 16
// of two on an SM, its shared memory as many as have room for the visited set: up to 65,536 centroids (8 KB) all of them, at 131,072 13
// blocks of two, from 262,144 on (32 KB) no more of two than of four, and then two warps leave an SM half as many to hide its
// latencies with.  A round of two-warp blocks takes about a third longer than one of four-warp blocks, which are fewer tokens.
// Measured (beam 32, 256 entries, four / two warps, us): 65,536 centroids: 1,184 tokens 164 / 212, 1,536 241 / 221, 8,192 834 / 718;
// 131,072: 1,536 290 / 278, 2,048 331 / 400, 4,096 562 / 579, 8,192 994 / 948; 262,144: 1,536 384 / 526, 8,192 1,550 / 2,091; a million:
// 8,192 6,574 / 9,556.  With 64 members and 512 entries the same sides win.
int graph_search_warps(const Index &ix, int64_t n_tokens)
{
    constexpr int64_t SM_SHARED = 228 * 1024, RESERVED = 1024;
    auto rounds = [&](int warps) {
        int64_t resident = 32 / warps;                       // __launch_bounds__
        if (visited_in_shared(ix)) {
            const int64_t room = SM_SHARED / ((ix.K + 31) / 32 * 4 + 2 * 4 * 32 * warps + 8 + RESERVED);
            if (resident > room) resident = room;
        }
        return (n_tokens + resident * ix.sm_count - 1) / (resident * ix.sm_count);
    };
    return 4 * rounds(2) < 3 * rounds(4) ? 2 : 4;
}

int check_graph_params(const Index &ix, const GraphSearch &g, int nprobe)
{
    if (!ix.graph) return fail(CHIMERA_INVALID_ARG, "the centroid graph is not built (chimera_index_build_graph)");
    if (g.beam < nprobe || g.beam > 64) return fail(CHIMERA_INVALID_ARG, "beam must be in [nprobe, 64], got %d", g.beam);
    if (g.n_entries < nprobe || g.n_entries > ix.K)
        return fail(CHIMERA_INVALID_ARG, "n_entries must be in [nprobe, n_centroids], got %d", g.n_entries);
    if (g.max_expansions < 0) return fail(CHIMERA_INVALID_ARG, "max_expansions must be >= 0");
    return CHIMERA_OK;
}

int launch_graph_probes(const Index &ix, const float *queries, int64_t n_tokens, int nprobe, const GraphSearch &g,
                        uint32_t *visited, bool want_visited, int32_t *out_probes, int32_t *out_scores, int32_t *out_nvis,
                        cudaStream_t st)
{
    const int64_t vwords = (ix.K + 31) / 32;
    const size_t smem = sizeof(uint32_t) * (size_t)vwords;
    const bool shared = visited_in_shared(ix);
    const bool wide = g.beam > 32, four = graph_search_warps(ix, n_tokens) == 4;
    auto kern = four ? (wide ? (shared ? graph_probe_kernel<true, true, 4> : graph_probe_kernel<false, true, 4>)
                             : (shared ? graph_probe_kernel<true, false, 4> : graph_probe_kernel<false, false, 4>))
                     : (wide ? (shared ? graph_probe_kernel<true, true, 2> : graph_probe_kernel<false, true, 2>)
                             : (shared ? graph_probe_kernel<true, false, 2> : graph_probe_kernel<false, false, 2>));
    if (shared) CHIMERA_CUDA(allow_shared(kern, VISITED_SMEM));
    else CHIMERA_CUDA(cudaMemsetAsync(visited, 0, graph_scratch_bytes(ix, n_tokens), st));
    launch(kern, (unsigned)n_tokens, four ? 128 : 64, shared ? smem : 0, st, queries, ix.D, ix.xc, ix.graph, ix.graph_deg, ix.K,
           g.n_entries, g.beam, g.max_expansions, nprobe, shared && !want_visited ? nullptr : visited, vwords, out_probes,
           out_scores, out_nvis);
    CHIMERA_CUDA(cudaGetLastError());
    count_launch(SLOT_PROBE, 1);
    return CHIMERA_OK;
}

}  // namespace chimera
