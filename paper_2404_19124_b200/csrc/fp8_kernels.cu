// Kernels of the reduced-precision vocabulary head (levels whose head GEMM is bound by reading the
// weights: fewer rows than the roofline ridge).  The head's weights exist a second time as e4m3 bytes
// with one scale per vocabulary row, half the bytes of the bf16 matrix.  Per level:
//   mix step            also writes the states as e4m3 (row_ops.cuh)
//   head GEMM           kind::f8f6f4 on the two e4m3 operands; the epilogue rescales the accumulators
//                       and keeps 8 candidates by APPROXIMATE logit and the (max, sum-exp) of the
//                       approximate logits: per vocabulary tile with the nodes as MMA rows, per CTA
//                       (all its vocabulary rows, 872 of 128256) with the nodes as columns
//   merge_rescore       folds those lists into a short list of max(8, 2 topk + 2), at most 16, tokens per
//                       row and the row's log-sum-exp, recomputes the short-listed logits EXACTLY from the
//                       bf16 weights and states (fp32 accumulation, as the bf16 head does), and takes
//                       the top-k of those
// The tokens and their logits are therefore those of the bf16 path whenever the true top-k are in the short
// list, which takes that no more than eight of its tokens lie in one list (the approximation error is a few
// hundredths of the logits' standard deviation; the k-th best of tens of thousands of logits and the last of the
// short list are much further apart); only the normaliser comes from approximate logits (error of order
// 1e-3, tolerance 2e-2).
#include "row_ops.cuh"

namespace spec {

namespace {

using namespace rows;

constexpr int kQuantThreads = 256;
constexpr int kRescoreThreads = 512;            // one warp per short-listed token
constexpr int kShortList = kRescoreThreads / 32;
static_assert(kShortList <= kMaxRounds, "scratch arrays");

// One CTA per row of X (bf16 [rows, d], d % 16 == 0): Q = e4m3(X / scale), scale = max|row| / 448.
__global__ void __launch_bounds__(kQuantThreads)
quantize_rows_kernel(const uint16_t *__restrict__ X, int d, uint8_t *__restrict__ Q, float *__restrict__ scale) {
    __shared__ float red[32];
    const size_t r = blockIdx.x;
    const uint16_t *x = X + r * d;
    float amax = 0.0f;
    for (int i = threadIdx.x * 8; i < d; i += kQuantThreads * 8) {
        const uint4 q = *(const uint4 *)(x + i);
        const uint32_t w[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
        for (int j = 0; j < 4; ++j)
            amax = fmaxf(amax, fmaxf(fabsf(__uint_as_float(w[j] << 16)), fabsf(__uint_as_float(w[j] & 0xffff0000u))));
    }
    const float s = row_scale_of(group_max<kQuantThreads, BlockSync>(amax, red, threadIdx.x));
    const float inv = 1.0f / s;
    for (int i = threadIdx.x * 8; i < d; i += kQuantThreads * 8) {
        const uint4 q = *(const uint4 *)(x + i);
        const uint32_t w[4] = {q.x, q.y, q.z, q.w};
        float v[8];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            v[2 * j] = __uint_as_float(w[j] << 16);
            v[2 * j + 1] = __uint_as_float(w[j] & 0xffff0000u);
        }
        *(uint2 *)(Q + r * d + i) = e4m3x8(v, inv);
    }
    if (threadIdx.x == 0) scale[r] = s;
}

struct RescoreArgs {
    MergeArgs merge;          // partial lists of approximate logits; tok_out / score_out: the children
    const uint16_t *W;        // bf16 [V, d] head weights
    const uint16_t *S;        // bf16 [rows, d] states of the level
    int d, V;
};

// Row r's children: the top-k of the exactly recomputed logits of its short list, written if `writer`.  Every warp finds
// them all; the token of child `pick` is returned to every thread.  `exact`: shared, kShortList floats.  `meanwhile`: see
// merge_select.
template <typename Meanwhile = Nothing>
__device__ __forceinline__ int rescore_row(const RescoreArgs &a, int r, int tid, Scratch *sc, float *exact, bool writer,
                                           int pick, Meanwhile meanwhile = Meanwhile()) {
    const int lane = tid & 31, warp = tid >> 5;
    const float base = (tid == 0 && a.merge.score_in) ? __ldcg(a.merge.score_in + r) : 0.0f;
    // short list: twice the branching factor plus two, at least 8, at most one per warp
    const int n_short = min(kShortList, max(8, 2 * a.merge.topk + 2));
    const MergeOut o = merge_select<kRescoreThreads, 8, BlockSync>(a.merge, r, tid, sc, n_short, meanwhile);
    const int short_id = o.id;   // lane j: the j-th short-listed token
    // exact logit of short-listed token `warp`: dot product of two bf16 rows, fp32 accumulation
    const int v = warp < n_short ? __shfl_sync(0xffffffffu, short_id, warp) : -1;
    float acc = 0.0f;
    if (v >= 0 && v < a.V) {
        const uint16_t *w = a.W + (size_t)v * a.d, *s = a.S + (size_t)r * a.d;
        constexpr int kBatch = 8;   // 8-element groups per lane whose loads are in flight together
        for (int i0 = lane * 8; i0 < a.d; i0 += 32 * 8 * kBatch) {
            uint4 qw[kBatch], qs[kBatch];
#pragma unroll
            for (int u = 0; u < kBatch; ++u) {
                const int i = i0 + u * 32 * 8;
                qw[u] = make_uint4(0u, 0u, 0u, 0u);
                qs[u] = qw[u];
                if (i < a.d) {
                    qw[u] = *(const uint4 *)(w + i);
                    qs[u] = __ldcg((const uint4 *)(s + i));
                }
            }
#pragma unroll
            for (int u = 0; u < kBatch; ++u) {
                const uint32_t ww[4] = {qw[u].x, qw[u].y, qw[u].z, qw[u].w}, ss[4] = {qs[u].x, qs[u].y, qs[u].z, qs[u].w};
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    acc = fmaf(__uint_as_float(ww[j] << 16), __uint_as_float(ss[j] << 16), acc);
                    acc = fmaf(__uint_as_float(ww[j] & 0xffff0000u), __uint_as_float(ss[j] & 0xffff0000u), acc);
                }
            }
        }
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, off);
    if (lane == 0) exact[warp] = (v >= 0 && v < a.V) ? acc : -INFINITY;
    __syncthreads();
    // the top-k of the exact logits, (value desc, token id asc)
    float val = lane < n_short ? exact[lane] : -INFINITY;
    int id = lane < n_short ? short_id : 0x7fffffff;
    const int topk = a.merge.topk;
    int picked = -1;
    for (int j = 0; j < topk; ++j) {
        const uint32_t key = float_key(val);
        const uint32_t bk = __reduce_max_sync(0xffffffffu, key);
        const uint32_t bi = __reduce_min_sync(0xffffffffu, key == bk ? (uint32_t)id : 0xffffffffu);
        if (j == pick) picked = (int)bi;
        if (writer && tid == 0) {
            a.merge.tok_out[(size_t)r * topk + j] = (int)bi;
            a.merge.score_out[(size_t)r * topk + j] = base + (key_float(bk) - o.lse);
        }
        if (warp == 0 && a.merge.next_emb != nullptr && bi < (uint32_t)a.merge.next_emb_rows) {   // (see prefetch_embeddings)
            const char *row = (const char *)a.merge.next_emb + (size_t)bi * a.merge.next_emb_bytes;
            for (int i = lane * 128; i < a.merge.next_emb_bytes; i += 32 * 128)
                asm volatile("prefetch.global.L2 [%0];" ::"l"(row + i));
        }
        if (key == bk && (uint32_t)id == bi) {   // taken
            val = -INFINITY;
            id = 0x7fffffff;
        }
    }
    return picked;
}

// One CTA per row.
__global__ void __launch_bounds__(kRescoreThreads) merge_rescore_kernel(RescoreArgs a) {
    extern __shared__ LeafKey rescore_keys[];   // prune_smem_bytes when the prune is folded in, else nothing
    __shared__ Scratch sc;
    __shared__ float exact[kShortList];
    __shared__ int last_of_sequence;
    griddep_launch();
    griddep_wait();
    rescore_row(a, blockIdx.x, threadIdx.x, &sc, exact, true, -1);
    prune_if_last<kRescoreThreads, BlockSync>(a.merge, blockIdx.x, threadIdx.x, rescore_keys, &last_of_sequence);
}

// One CTA per child, up to one per SM: re-scores its parent's short list (the siblings find the weight rows in L2) and
// computes the child's state, as merge_mix_child_kernel does for bf16 heads.  One launch, one barrier between grids and one
// round trip of the token through memory less per level: the 13B step with e4m3 heads 243 -> 240 us, two levels of 60
// nodes 88.3 -> 87.2, 16 sequences times 8 nodes 96.1 -> 94.3.  More children than SMs would take turns on them.
struct RescoreMixArgs {
    RescoreArgs rescore;
    MixArgs mix;
};
__global__ void __maxnreg__(72) rescore_mix_child_kernel(RescoreMixArgs a) {
    __shared__ Scratch sc;
    __shared__ float exact[kShortList], red[2 * kMaxGroupWarps];
    griddep_launch();
    griddep_wait();
    const int c = blockIdx.x, topk = a.rescore.merge.topk, r = c / topk;
    float pre[1][8];
    const int t = rescore_row(a.rescore, r, threadIdx.x, &sc, exact, c == r * topk, c - r * topk,
                              [&] { parent_state<kRescoreThreads>(a.mix, r, threadIdx.x, pre); });
    mix_ln_gelu_row<kRescoreThreads, 1, 1, BlockSync>(a.mix, c, r, t, threadIdx.x, red, pre);
}

}  // namespace

int launch_quantize_rows(const void *X, int rows, int d, void *Q, float *scale, cudaStream_t st) {
    if (rows <= 0 || d <= 0 || d % 16 != 0) return SPEC_ERR_SHAPE;
    quantize_rows_kernel<<<rows, kQuantThreads, 0, st>>>((const uint16_t *)X, d, (uint8_t *)Q, scale);
    SPEC_CUDA_TRY(cudaGetLastError());
    return SPEC_OK;
}

int launch_merge_rescore(const MergeArgs &g, const void *W, const void *S, int rows, int d, int V, cudaStream_t st) {
    RescoreArgs a{};
    a.merge = g;
    a.W = (const uint16_t *)W;
    a.S = (const uint16_t *)S;
    a.d = d;
    a.V = V;
    const size_t smem = g.seq_done ? prune_smem_bytes(g.L, g.Lpad) : 0;
    SPEC_CUDA_TRY(launch_pdl(merge_rescore_kernel, dim3(rows), dim3(kRescoreThreads), smem, st, a));
    return SPEC_OK;
}

int launch_rescore_mix(const MergeArgs &g, const void *W, const void *S, const MixArgs &m, int rows, int d, int V,
                       cudaStream_t st) {
    if (m.d > 8 * kRescoreThreads || rows * g.topk > num_sms() || g.seq_done != nullptr) return SPEC_ERR_SHAPE;
    RescoreMixArgs a{};
    a.rescore.merge = g;
    a.rescore.merge.next_emb = nullptr;   // the gather follows in the same CTA
    a.rescore.W = (const uint16_t *)W;
    a.rescore.S = (const uint16_t *)S;
    a.rescore.d = d;
    a.rescore.V = V;
    a.mix = m;
    SPEC_CUDA_TRY(launch_pdl(rescore_mix_child_kernel, dim3(rows * g.topk), dim3(kRescoreThreads), 0, st, a));
    return SPEC_OK;
}

}  // namespace spec
