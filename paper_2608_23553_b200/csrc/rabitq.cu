// The paper's GPU pipeline on RaBitQ 1-bit codes (Sec. 2.2 for the codec, Sec. 3.2 steps 2 and 3 for its use):
//   q_p = P q                                         (rotation; inner products are preserved)
//   est(i, t) = <q_p, o_p-bar> / <o_p, o_p-bar>,  <q_p, o_p-bar> = (1 / |y-bar|) (<q_p, o_b> - 1/2 sum q_p)
// evaluated as  inv_dot_t * (c * (float)(2 T - SQ_i)),  T = sum_x Xq_i[x] o_b[x],  SQ_i = sum_x Xq_i[x],
// Xq = rint(q_p * 2^22),  c = 1 / (sqrt(D) 2^22): integers plus two fp32 multiplications in a fixed order, and sums
// over query tokens in increasing order, so every result is reproducible bit for bit.
//
// This file: attaching the codes to an index, the rotation kernel, and candidate refinement by partial 1-bit scores
// (Algorithm 2; a block per (query token, posting list) as in the paper's design; the maxima of Algorithm 4 as visit
// lists for batches on large corpora, g3_visits.cuh, otherwise a table of rows updated with atomicMax).
// The complete 1-bit scores of the survivors run on the tensor cores (g4_residual_umma.cu, RQ variant).
#include <math.h>

#include "g3_visits.cuh"

namespace chimera {

__global__ void transpose_kernel(const float *__restrict__ in, int D, float *__restrict__ out)
{
    int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e < D * D) {
        int r = e / D, x = e % D;
        out[x * D + r] = in[e];
    }
}

int transpose_rotation(const Index &ix, const float *rotation, float **rot_t, cudaStream_t st)
{
    *rot_t = nullptr;
    float *out = nullptr;
    CHIMERA_CUDA(cudaMalloc(&out, sizeof(float) * ix.D * ix.D));
    transpose_kernel<<<(ix.D * ix.D + 255) / 256, 256, 0, st>>>(rotation, ix.D, out);
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) {
        cudaFree(out);
        return fail(CHIMERA_CUDA_ERROR, "rotation: %s", cudaGetErrorString(e));
    }
    *rot_t = out;
    return CHIMERA_OK;
}

// grid (B * nq), block D: q_p[row][r] = sum_x P[r][x] q[row][x] as one fma chain in increasing x.
__global__ void __launch_bounds__(128)
rotate_kernel(const float *__restrict__ rot_t, const float *__restrict__ q, int D, float *__restrict__ out)
{
    pdl_entry();
    __shared__ float qrow[128];
    const int64_t row = blockIdx.x;
    const int r = threadIdx.x;
    if (r < D) qrow[r] = q[row * D + r];
    __syncthreads();
    if (r < D) {
        float acc = 0.0f;
        for (int x = 0; x < D; ++x) acc = fmaf(rot_t[x * D + r], qrow[x], acc);
        out[row * D + r] = acc;
    }
}

int launch_rotate(const Index &ix, const Params &p, const float *queries, float *q_rot, cudaStream_t st)
{
    launch(rotate_kernel, (unsigned)((int64_t)p.B * p.nq), 128, 0, st, ix.rot_t, queries, ix.D, q_rot);
    CHIMERA_CUDA(cudaGetLastError());
    count_launch(SLOT_G1);
    return CHIMERA_OK;
}

constexpr int RP_THREADS = 128;

// grid (blocks, B): zero the first n_cand[b] rows of M.
__global__ void __launch_bounds__(256)
rabitq_clear_kernel(int32_t *__restrict__ M, const int32_t *__restrict__ n_cand, int64_t maxc, int nq)
{
    pdl_entry();
    const int b = blockIdx.y;
    const int64_t n = (int64_t)n_cand[b] * nq;
    int32_t *row = M + (int64_t)b * maxc * nq;
    const int64_t tid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, stride = (int64_t)gridDim.x * blockDim.x;
    if ((nq & 3) == 0) {                               // rows are 16-byte aligned
        int4 *row4 = reinterpret_cast<int4 *>(row);
        for (int64_t e = tid; e < n / 4; e += stride) row4[e] = make_int4(0, 0, 0, 0);
    } else {
        for (int64_t e = tid; e < n; e += stride) row[e] = 0;
    }
}

// grid (nq * splits, B): lists p, p + splits, ... of a query token per block; M holds float bits (>= 0, so integer order =
// float order).  bits / inv_dot: in list order (tok_id NULL), or the caller's document-major arrays.
template <bool LISTS>
__global__ void __launch_bounds__(RP_THREADS)
rabitq_partial_kernel(const int8_t *__restrict__ qdig, int nq, int B, int CW, int P, float c,
                      const int32_t *__restrict__ probes, const int64_t *__restrict__ tok_off,
                      const int32_t *__restrict__ tok_id, const int32_t *__restrict__ tok_doc,
                      const uint32_t *__restrict__ bits, const float *__restrict__ inv_dot,
                      const uint2 *__restrict__ ranks, int64_t words, int64_t maxc, int32_t *__restrict__ M,
                      VisitLists lists, int64_t longest, int splits)
{
    pdl_entry();
    __shared__ __align__(16) QueryDigits dig;
    const int b = blockIdx.y;
    const int i = blockIdx.x / splits;
    load_query_digits(dig, qdig, (int64_t)B * residual_rows(nq), (int64_t)b * residual_rows(nq) + score_row(i));
    __syncthreads();
    const int sq = query_sum(dig);
    const uint2 *rk = ranks + (int64_t)b * words;
    int32_t *Mb = LISTS ? nullptr : M + (int64_t)b * maxc * nq;
    unsigned long long *heads = LISTS ? lists.head + (int64_t)b * maxc : nullptr;
    unsigned long long *nodes = LISTS ? lists.node + (int64_t)b * lists.cap : nullptr;
    uint32_t v0;                                       // node of the list's first entry
    int64_t e0;
    // (the token's factor, the document's bitmap word and its rank come as arguments: they depend on the list entry
    // alone, so their loads are issued with the code loads instead of one after the other behind the score)
    VisitPush push[2];
    auto update = [&](int n, int64_t e, uint32_t d, float factor, int T, uint2 r) {
        const float est = __fmul_rn(factor, __fmul_rn(c, (float)(2 * T - sq)));
        if (est > 0.0f) {                              // the table starts at 0 (Algorithm 2)
            const int64_t rank = (int64_t)r.y + __popc(r.x & ((1u << (d & 31)) - 1u));
            if (rank < maxc && DBG_RANK_OK(rank)) {
                if (LISTS) visit_begin(push[n], heads + rank, v0 + (uint32_t)(e - e0), i, __float_as_uint(est));
                else atomicMax(&Mb[rank * nq + i], __float_as_int(est));
            }
        }
    };
    for (int p = blockIdx.x % splits; p < P; p += splits) {
        const int32_t cen = DBG_CID(probes[((int64_t)b * nq + i) * P + p]);
        v0 = (uint32_t)((i * P + p) * longest);
        e0 = tok_off[cen];
        const int64_t e1 = tok_off[cen + 1];
        // two visits per thread and iteration, their loads issued together (the second one past the end repeats the first)
        for (int64_t e = e0 + threadIdx.x; e < e1; e += 2 * RP_THREADS) {
            const int64_t at[2] = {e, e + RP_THREADS < e1 ? e + RP_THREADS : e};
            uint32_t d[2], w[2][CODE_WORDS<1>];
            uint2 r[2];
            float f[2];
#pragma unroll
            for (int n = 0; n < 2; ++n) {
                const int64_t t = DBG_TOK(tok_id ? (int64_t)tok_id[at[n]] : at[n]);
                load_code<1>(w[n], bits + t * CW, CW);
                f[n] = __ldg(inv_dot + t);
                d[n] = (uint32_t)DBG_DOC(tok_doc[at[n]]);
                r[n] = __ldg(rk + (d[n] >> 5));
            }
            if (LISTS) { visit_end(push[0], nodes); visit_end(push[1], nodes); }
            int T[2];
            code_dots<1, 2>(T, w, CW, dig);
            update(0, at[0], d[0], f[0], T[0], r[0]);
            if (at[1] != e) update(1, at[1], d[1], f[1], T[1], r[1]);
        }
    }
    if (LISTS) { visit_end(push[0], nodes); visit_end(push[1], nodes); }
}

// grid (blocks, B): F'[b][j] = M[b][j][0] + M[b][j][1] + ... in that order (fp32), one thread per candidate.
__global__ void __launch_bounds__(256)
rabitq_sum_kernel(const int32_t *__restrict__ M, const int32_t *__restrict__ n_cand, int64_t maxc, int nq,
                  int32_t *__restrict__ fprime_bits)
{
    pdl_entry();
    const int b = blockIdx.y;
    const int n = n_cand[b];
    for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < n; j += gridDim.x * blockDim.x) {
        const int32_t *row = M + ((int64_t)b * maxc + j) * nq;
        float s = 0.0f;
        if ((nq & 3) == 0) {
            const int4 *row4 = reinterpret_cast<const int4 *>(row);
            for (int i = 0; i < nq / 4; ++i) {
                const int4 v = row4[i];
                s = __fadd_rn(s, __int_as_float(v.x));
                s = __fadd_rn(s, __int_as_float(v.y));
                s = __fadd_rn(s, __int_as_float(v.z));
                s = __fadd_rn(s, __int_as_float(v.w));
            }
        } else {
            for (int i = 0; i < nq; ++i) s = __fadd_rn(s, __int_as_float(row[i]));
        }
        fprime_bits[(int64_t)b * maxc + j] = __float_as_int(s);
    }
}

int launch_rabitq_partial(const Index &ix, const Params &p, const Layout &L, const int8_t *qdig_rot,
                          const int32_t *probes, const uint2 *ranks, const int32_t *n_cand, void *partial_m,
                          int32_t *fprime_bits, cudaStream_t st)
{
    const bool use_lists = L.visit_nodes > 0;
    const VisitLists lists = visit_lists(p, L, partial_m);
    int32_t *M = (int32_t *)partial_m;
    const dim3 gclr((unsigned)(((int64_t)ix.sm_count * 8 + p.B - 1) / p.B), (unsigned)p.B);
    int rc;
    if (use_lists) {
        if ((rc = launch_visit_clear(ix, p, lists, n_cand, st))) return rc;
    } else {
        launch(rabitq_clear_kernel, gclr, 256, 0, st, M, n_cand, p.maxc, p.nq);
        CHIMERA_CUDA(cudaGetLastError());
    }
    const float c = (float)(1.0 / (sqrt((double)ix.D) * 4194304.0));
    const int splits = refine_splits(ix, p);
    const dim3 grid((unsigned)(p.nq * splits), (unsigned)p.B);
    const uint32_t *bits = reinterpret_cast<const uint32_t *>(ix.list_bits ? ix.list_bits : ix.rq_bits);
    const float *inv = ix.list_bits ? ix.list_inv : ix.rq_inv;
    const int32_t *ids = ix.list_bits ? nullptr : ix.tok_id;
    if (use_lists)
        launch(rabitq_partial_kernel<true>, grid, RP_THREADS, 0, st, qdig_rot, p.nq, p.B, ix.D / 32, p.P, c, probes, ix.tok_off, ids,
                                                                 ix.tok_doc, bits, inv, ranks, L.words, p.maxc, M,
                                                                 lists, ix.max_tok_list, splits);
    else
        launch(rabitq_partial_kernel<false>, grid, RP_THREADS, 0, st, qdig_rot, p.nq, p.B, ix.D / 32, p.P, c, probes, ix.tok_off, ids,
                                                                  ix.tok_doc, bits, inv, ranks, L.words, p.maxc, M,
                                                                  lists, ix.max_tok_list, splits);
    CHIMERA_CUDA(cudaGetLastError());
    if (use_lists) {
        if ((rc = launch_visit_sum(ix, p, lists, true, n_cand, fprime_bits, st))) return rc;
    } else {
        launch(rabitq_sum_kernel, gclr, 256, 0, st, M, n_cand, p.maxc, p.nq, fprime_bits);
        CHIMERA_CUDA(cudaGetLastError());
    }
    count_launch(SLOT_CI, 3);
    return CHIMERA_OK;
}

}  // namespace chimera
