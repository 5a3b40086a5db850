// Stand-alone row kernels of the draft path (the row-wise steps themselves are in row_ops.cuh):
//   mix_ln_gelu_kernel   one CTA of 256 threads per tree node
//   merge_expand_kernel  one CTA of 160 threads per row of the vocabulary head
//   prune_kernel         one CTA of 256 threads per sequence
//   merge_prune_kernel   one CTA per sequence, one warp per row: the last level's merge and the prune in one
// Each is launched with programmatic stream serialization, so its CTAs are usually resident, waiting,
// while the kernel before it still runs.
#include "row_ops.cuh"

namespace spec {

namespace {

using namespace rows;

constexpr int kRowThreads = 256;
constexpr int kFusedChildren = 2;   // of a row, in merge_mix_kernel
constexpr int kMergeThreads = 160;   // one list per thread up to V = 35000 (a CTA of the head GEMM leaves one)

// Rows of up to 2048 elements: at most 128 registers, so that two CTAs fit beside a resident GEMM CTA.
__global__ void __launch_bounds__(kRowThreads, 2) mix_ln_gelu_kernel(MixArgs m) {
    __shared__ float red[32];
    griddep_launch();
    griddep_wait();
    const int r = blockIdx.x, t = __ldcg(m.tok + r);
    mix_ln_gelu_row<kRowThreads, 1, 2, BlockSync>(m, r, r / m.parent_div, t, threadIdx.x, red);
}

// Rows of 2049 to 4096 elements in levels of at most one CTA per SM: 512 threads, one 8-element group each.  The
// step is a chain of dependent latencies (loads, two reductions, sixteen erf evaluations per thread with 256
// threads), so halving the per-thread work shortens it: 13B-shaped draft 3-5 us faster than with 256 threads.  At
// most 72 registers, so that the CTA fits beside a resident GEMM CTA.
constexpr int kWideRowThreads = 512;
__global__ void __maxnreg__(72) mix_ln_gelu_512_kernel(MixArgs m) {
    __shared__ float red[32];
    griddep_launch();
    griddep_wait();
    const int r = blockIdx.x, t = __ldcg(m.tok + r);
    mix_ln_gelu_row<kWideRowThreads, 1, 1, BlockSync>(m, r, r / m.parent_div, t, threadIdx.x, red);
}

// The same for levels with more nodes than one wave of the kernel above holds: one 8-element group in
// flight per thread and at most 80 registers, so three CTAs share an SM and the level stays one wave.
__global__ void __launch_bounds__(kRowThreads, 3) mix_ln_gelu_many_kernel(MixArgs m) {
    __shared__ float red[32];
    griddep_launch();
    griddep_wait();
    const int r = blockIdx.x, t = __ldcg(m.tok + r);
    if (m.d <= 8 * kRowThreads) mix_ln_gelu_row<kRowThreads, 1, 1, BlockSync>(m, r, r / m.parent_div, t, threadIdx.x, red);
    else mix_ln_gelu_row<kRowThreads, 2, 1, BlockSync>(m, r, r / m.parent_div, t, threadIdx.x, red);
}

// Levels of several waves whose projection was not split (more than 128 parents, or too few K blocks): throughput counts, and
// a CTA has only as many threads as its row needs with two groups each.  2016 rows of 400 elements 14.7 -> 6.9 us, 1836 of
// 2296 25.5 -> 21.5.  (Four rows to a CTA, or 128 threads with four groups each, are no better.)
// The only one of the separate kernels that takes the LayerNorm sums in order (launch_mix_ln_gelu).
__global__ void __launch_bounds__(kRowThreads, 3) mix_ln_gelu_waves_kernel(MixArgs m) {
    __shared__ float red[32];
    griddep_launch();
    griddep_wait();
    const int r = blockIdx.x, t = __ldcg(m.tok + r);
    mix_ln_gelu_row<0, 2, 1, BlockSync, 1>(m, r, r / m.parent_div, t, threadIdx.x, red, nullptr, m.in_order != 0);
}

// Rows of up to 16384 elements.
__global__ void __launch_bounds__(kRowThreads) mix_ln_gelu_mid_kernel(MixArgs m) {
    __shared__ float red[32];
    griddep_launch();
    griddep_wait();
    const int r = blockIdx.x, t = __ldcg(m.tok + r);
    if (m.d <= 8 * kRowThreads * 4) mix_ln_gelu_row<kRowThreads, 4, 2, BlockSync>(m, r, r / m.parent_div, t, threadIdx.x, red);
    else mix_ln_gelu_row<kRowThreads, 8, 2, BlockSync>(m, r, r / m.parent_div, t, threadIdx.x, red);
}

// Rows wider than the register version covers: the mixed row is staged in shared memory.
__global__ void __launch_bounds__(kRowThreads) mix_ln_gelu_wide_kernel(MixArgs m) {
    extern __shared__ float h_s[];   // [d]
    __shared__ float red[32];
    griddep_launch();
    griddep_wait();
    const int r = blockIdx.x, tid = threadIdx.x, d = m.d;
    const int t = m.tok[r];
    const bool tok_ok = (t >= 0) && (t < m.V);
    if (!tok_ok && tid == 0) report_error(m.err, SPEC_ERR_TOKEN_RANGE);
    const float *p = m.P + (size_t)(r / m.parent_div) * d;
    const uint16_t *e = m.emb + (size_t)(tok_ok ? t : 0) * d;
    float sum = 0.0f;
    for (int i = tid; i < d; i += kRowThreads) {
        float pv = 0.0f;
        for (int sp = 0; sp < m.p_splits; ++sp) pv += p[sp * m.p_split_stride + i];
        const float z = tok_ok ? bf16_bits_to_float(e[i]) : 0.0f;
        const float h = m.a * pv + m.b * z;
        h_s[i] = h;
        sum += h;
    }
    const float mean = group_sum<kRowThreads, BlockSync>(sum, red, tid) / (float)d;
    float sq = 0.0f;
    for (int i = tid; i < d; i += kRowThreads) {
        const float c = h_s[i] - mean;
        sq += c * c;
    }
    const float var = group_sum<kRowThreads, BlockSync>(sq, red + kMaxGroupWarps, tid) / (float)d;
    const float rstd = rsqrtf(var + m.eps);
    for (int i = tid; i < d; i += kRowThreads)
        m.S_out[(size_t)r * d + i] = (uint16_t)float_to_bf16_bits(gelu_erf((h_s[i] - mean) * rstd * m.gamma[i] + m.beta[i]));
}

// First kernel of a draft: clears the workspace header (error word, per-sequence counters).  A kernel
// rather than a memset so that the projection launched behind it may already set itself up and fetch
// weights; like every kernel here it first waits for whatever precedes it in the stream.
__global__ void __launch_bounds__(256) draft_init_kernel(int32_t *hdr, int words) {
    griddep_launch();
    griddep_wait();
    for (int i = threadIdx.x; i < words; i += blockDim.x) hdr[i] = 0;
}

template <int kLen>
__global__ void __launch_bounds__(kMergeThreads) merge_expand_kernel(MergeArgs g) {
    extern __shared__ LeafKey merge_keys[];   // prune_smem_bytes when the prune is folded in, else nothing
    __shared__ Scratch sc;
    __shared__ int last_of_sequence;
    griddep_launch();
    griddep_wait();
    merge_expand_row<kMergeThreads, kLen, BlockSync>(g, blockIdx.x, threadIdx.x, &sc);
    prune_if_last<kMergeThreads, BlockSync>(g, blockIdx.x, threadIdx.x, merge_keys, &last_of_sequence);
}

// The last level's merge and the prune, one CTA per sequence, one warp per row: the leaves' scores meet in shared memory, where
// with a CTA per row the rows of a sequence are counted in (a fence, an atomic, the scores back from L2: 3.4 us) and 384 CTAs take
// turns on the SMs.  A warp needs longer for a row than five (1.9 us for 143 lists), about 0.2 us per 32 lists beyond the first.
// Exposed time, a CTA per row -> this: 12 rows a sequence (7B shape) 6.2 -> 4.7 us, 24 rows of 16 sequences (13B) 9.0 -> 8.2; the
// batch-1 draft 129.5 -> 126.5, the ragged step 119.8 -> 118.3.
// At most 48 registers, so that the widest CTA fits beside a resident GEMM CTA.
struct OneWarp {
    static __device__ __forceinline__ void sync() { __syncwarp(); }
};
constexpr int kPruneRows = 24;   // rows of a sequence, at most: warps of the CTA
template <int kLen>
__global__ void __maxnreg__(48) merge_prune_kernel(MergeArgs g) {
    __shared__ float4 scores4[kPruneRows * SPEC_MAX_TOPK / 4];
    __shared__ int toks[kPruneRows * SPEC_MAX_TOPK];
    float *scores = (float *)scores4;
    griddep_launch();
    griddep_wait();
    const int b = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, L = g.L, topk = g.topk;
    const int r = b * g.rows_per_seq + warp;
    const float base = (lane < topk && g.score_in) ? __ldcg(g.score_in + r) : 0.0f;
    int32_t path[SPEC_MAX_HEADS];
    const MergeOut o = merge_select<32, kLen, OneWarp>(g, r, lane, nullptr, topk);
    // the ancestors of leaf `tid`, whose place depends on nothing but its index, on their way until the scores are there
    if (tid < L) {
        int idx = tid / topk, per_seq = g.rows_per_seq;
#pragma unroll
        for (int l = SPEC_MAX_HEADS - 2; l >= 0; --l) {
            if (l < g.prune.n - 1) {
                path[l] = __ldcg(g.prune.tok[l] + (size_t)b * per_seq + idx);
                idx /= g.prune.topk[l];
                per_seq /= g.prune.topk[l];
            }
        }
    }
    if (lane < topk) {
        const float score = base + (o.val - o.lse);
        g.tok_out[(size_t)r * topk + lane] = o.id;
        g.score_out[(size_t)r * topk + lane] = score;
        scores[warp * topk + lane] = score;
        toks[warp * topk + lane] = o.id;
    }
    if (tid < 3 && L + tid < (L + 3) / 4 * 4) scores[L + tid] = __int_as_float(0x7fffffff);   // (NaN: before nobody)
    __syncthreads();
    if (tid >= L) return;
    const float mine = scores[tid];
    int rank = 0;   // leaves before this one: a better score, or the same and a lower index
    for (int j = 0; j < L; j += 4) {
        const float4 s = scores4[j / 4];
        rank += (s.x > mine) | ((s.x == mine) & (j < tid));
        rank += (s.y > mine) | ((s.y == mine) & (j + 1 < tid));
        rank += (s.z > mine) | ((s.z == mine) & (j + 2 < tid));
        rank += (s.w > mine) | ((s.w == mine) & (j + 3 < tid));
    }
    if (rank >= g.K) return;
    const size_t c = (size_t)b * g.K + rank;
    g.cand_logp[c] = mine;
    int32_t *cand = g.cand_tok + c * g.prune.n;
#pragma unroll
    for (int l = 0; l < SPEC_MAX_HEADS - 1; ++l)
        if (l < g.prune.n - 1) cand[l] = path[l];
    cand[g.prune.n - 1] = toks[tid];
}

// Merge of level l and the gather + mix + LayerNorm + GELU of level l + 1 in one launch, for two children per row where there
// are more children than SMs but no more rows: one CTA of 256 threads per row of level l folds the row's partial lists into its
// children (tokens, scores) and then computes the states of those children, whose tokens it has just found and whose parent
// projection is this row's.  One kernel boundary less between two vocabulary heads.  75 / 128 / 148 rows, V 8000, the whole
// draft as two kernels -> this: d 1024 52.9 -> 51.4 us, 59.4 -> 56.7, 56.8 -> 54.5; d 2048 64.6 -> 62.8, 71.2 -> 68.4, 76.4 ->
// 74.5.
struct MergeMixArgs {
    MergeArgs merge;   // level l
    MixArgs mix;       // level l + 1 (tok and parent_div unused: the tokens come from the merge)
};

// At most 128 registers: like the other row kernels its CTAs must fit beside a resident GEMM CTA, or they could
// not start (and wait, set up) before that kernel ends.
__global__ void __launch_bounds__(kRowThreads, 2) merge_mix_kernel(MergeMixArgs a) {
    __shared__ Scratch sc;
    __shared__ float red_a[kRowThreads / 32 * kFusedChildren], red_b[kRowThreads / 32 * kFusedChildren];
    griddep_launch();
    griddep_wait();
    const int r = blockIdx.x, tid = threadIdx.x;
    const int tok = merge_expand_row<kRowThreads, list_slots(kFusedChildren), BlockSync>(a.merge, r, tid, &sc).id;
    mix_children<kRowThreads, 1, kFusedChildren, BlockSync>(a.mix, r, r * kFusedChildren, tok, red_a, red_b, tid);
}

// Rows of 2049 to 4096 elements: 512 threads, one 8-element group each, like mix_ln_gelu_512_kernel (d 4096, V 8000, 75 / 128 /
// 148 rows: 93.3 -> 91.1 us, 102.3 -> 98.1, 125.0 -> 122.0; V 32000 195.8 -> 192.0, 205.0 -> 203.7, 277.3 -> 274.1).  72 registers
// at most, so that the CTA fits beside a resident GEMM CTA.
__global__ void __maxnreg__(72) merge_mix_512_kernel(MergeMixArgs a) {
    __shared__ Scratch sc;
    __shared__ float red_a[kWideRowThreads / 32 * kFusedChildren], red_b[kWideRowThreads / 32 * kFusedChildren];
    griddep_launch();
    griddep_wait();
    const int r = blockIdx.x, tid = threadIdx.x;
    const int tok = merge_expand_row<kWideRowThreads, list_slots(kFusedChildren), BlockSync>(a.merge, r, tid, &sc).id;
    mix_children<kWideRowThreads, 1, kFusedChildren, BlockSync>(a.mix, r, r * kFusedChildren, tok, red_a, red_b, tid);
}

// The same with one CTA per CHILD, for levels whose children are at most one per SM: every child's CTA repeats its
// parent's merge (a few KB from L2) and computes its own state, so no parallelism is lost and a kernel boundary is saved.
// Levels 0 -> 1 -> 2 of the 7B shape (8 -> 32 -> 96 nodes): 10.2 us a level as two kernels, 8.0 as one; the step 160.8 ->
// 158.9 us, smallest shape 51.2 -> 48.4, ragged step 131.2 -> 129.3, single-candidate chain 163.6 -> 161.5.
// With one or two children per row the LayerNorm sums are added in the order of merge_mix_kernel, which takes such levels beyond
// one child per SM, so that a level's states are the same bits on both sides of that line.  (In a tree a sum's last bit
// differs, now and then a state rounds to the other bf16 neighbour and a score moves by up to 1e-3.)
template <int kThreads, int kLen>
__device__ __forceinline__ void merge_mix_child(const MergeMixArgs &a, Scratch *sc, float *red) {
    const int c = blockIdx.x, topk = a.merge.topk, r = c / topk, tid = threadIdx.x;
    float pre[1][8];
    const MergeOut o = merge_expand_row<kThreads, kLen, BlockSync>(a.merge, r, tid, sc, c == r * topk,
                                                                   [&] { parent_state<kThreads>(a.mix, r, tid, pre); });
    const int t = __shfl_sync(0xffffffffu, o.id, c - r * topk);
    const bool in_order = topk <= kFusedChildren && a.mix.S8_out == nullptr;
    mix_ln_gelu_row<kThreads, 1, 1, BlockSync>(a.mix, c, r, t, tid, red, pre, in_order);
}
template <int kLen>
__global__ void __launch_bounds__(kRowThreads, 2) merge_mix_child_kernel(MergeMixArgs a) {
    __shared__ Scratch sc;
    __shared__ float red[32];
    griddep_launch();
    griddep_wait();
    merge_mix_child<kRowThreads, kLen>(a, &sc, red);
}
template <int kLen>
__global__ void __maxnreg__(72) merge_mix_child_512_kernel(MergeMixArgs a) {
    __shared__ Scratch sc;
    __shared__ float red[32];
    griddep_launch();
    griddep_wait();
    merge_mix_child<kWideRowThreads, kLen>(a, &sc, red);
}

// Vocabulary-parallel head: one warp per row folds the n_ranks raw lists (see launch_merge_shards).
// Lane i owns entries i and i + 32 of the row's n_ranks * topk <= 64 candidates.
constexpr int kShardRowsPerCta = 4;
__global__ void __launch_bounds__(32 * kShardRowsPerCta)
merge_shards_kernel(const char *slots, size_t slot_bytes, int n_ranks, int rows, int topk,
                    const float *__restrict__ score_in, int32_t *__restrict__ tok_out, float *__restrict__ score_out) {
    griddep_launch();
    griddep_wait();
    const int lane = threadIdx.x & 31;
    const int r = blockIdx.x * kShardRowsPerCta + (threadIdx.x >> 5);
    if (r >= rows) return;
    const int n_cand = n_ranks * topk;
    float v[2];
    int id[2];
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        const int c = lane + 32 * q;
        v[q] = -INFINITY;
        id[q] = 0x7fffffff;
        if (c < n_cand) {
            const int g = c / topk, j = c - g * topk;
            const char *slot = slots + (size_t)g * slot_bytes;
            const float *val = reinterpret_cast<const float *>(slot);
            const int32_t *tok = reinterpret_cast<const int32_t *>(slot + sizeof(float) * (size_t)rows * topk);
            v[q] = __ldcg(val + (size_t)r * topk + j);
            id[q] = __ldcg(tok + (size_t)r * topk + j);
        }
    }
    // log-sum-exp over the whole vocabulary from the shards' values, lane g holding shard g
    float l = -INFINITY;
    if (lane < n_ranks) {
        const char *slot = slots + (size_t)lane * slot_bytes;
        l = __ldcg(reinterpret_cast<const float *>(slot + 2 * sizeof(float) * (size_t)rows * topk) + r);
    }
    float m = l;
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, off));
    float e = (lane < n_ranks && l > -INFINITY) ? expf(l - m) : 0.0f;
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) e += __shfl_xor_sync(0xffffffffu, e, off);
    const float lse = m + logf(e);
    const float base = score_in ? __ldcg(score_in + r) : 0.0f;
    for (int j = 0; j < topk; ++j) {
        // the lane's better entry, then the warp's best: (value desc, token id asc)
        const int mine = better(v[1], id[1], v[0], id[0]) ? 1 : 0;
        const uint32_t key = float_key(v[mine]);
        const uint32_t bk = __reduce_max_sync(0xffffffffu, key);
        const uint32_t bi = __reduce_min_sync(0xffffffffu, key == bk ? (uint32_t)id[mine] : 0xffffffffu);
        if (lane == 0) {
            tok_out[(size_t)r * topk + j] = (int)bi;
            score_out[(size_t)r * topk + j] = base + (key_float(bk) - lse);
        }
        if (key == bk && (uint32_t)id[mine] == bi) {   // token ids are unique across shards: one owner
            v[mine] = -INFINITY;
            id[mine] = 0x7fffffff;
        }
    }
}

__global__ void __launch_bounds__(kRowThreads)
prune_kernel(const float *leaf_score, PruneArgs pa, int L, int Lpad, int K, int32_t *cand_tok, float *cand_logp) {
    extern __shared__ LeafKey keys[];   // prune_smem_bytes
    griddep_launch();
    griddep_wait();
    prune_sequence<kRowThreads, BlockSync>(leaf_score, pa, L, Lpad, K, cand_tok, cand_logp, blockIdx.x, threadIdx.x,
                                           keys);
}

}  // namespace

int launch_mix_ln_gelu(const MixArgs &m, int rows, cudaStream_t st) {
    const int d_inner = m.d;
    // (in_order: set only behind more parents than SMs, whose projection is not split where there are 128 SMs or more)
    if (d_inner <= 8 * kRowThreads * 2 && rows > num_sms() && (m.p_splits == 1 || m.in_order)) {
        SPEC_CUDA_TRY(launch_pdl(mix_ln_gelu_waves_kernel, dim3(rows), dim3((d_inner + 511) / 512 * 32), 0, st, m));
    } else if (d_inner <= 8 * kRowThreads * 2 && rows > num_sms()) {
        SPEC_CUDA_TRY(launch_pdl(mix_ln_gelu_many_kernel, dim3(rows), dim3(kRowThreads), 0, st, m));
    } else if (d_inner <= 8 * kRowThreads) {
        SPEC_CUDA_TRY(launch_pdl(mix_ln_gelu_kernel, dim3(rows), dim3(kRowThreads), 0, st, m));
    } else if (d_inner <= 8 * kWideRowThreads) {
        SPEC_CUDA_TRY(launch_pdl(mix_ln_gelu_512_kernel, dim3(rows), dim3(kWideRowThreads), 0, st, m));
    } else if (d_inner <= 8 * kRowThreads * 8) {
        SPEC_CUDA_TRY(launch_pdl(mix_ln_gelu_mid_kernel, dim3(rows), dim3(kRowThreads), 0, st, m));
    } else {
        const size_t smem = sizeof(float) * (size_t)d_inner;
        if (smem > 48 * 1024)
            SPEC_CUDA_TRY(cudaFuncSetAttribute(mix_ln_gelu_wide_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                               (int)smem));
        SPEC_CUDA_TRY(launch_pdl(mix_ln_gelu_wide_kernel, dim3(rows), dim3(kRowThreads), smem, st, m));
    }
    return SPEC_OK;
}

int launch_draft_init(int32_t *hdr, int words, cudaStream_t st) {
    SPEC_CUDA_TRY(launch_pdl(draft_init_kernel, dim3(1), dim3(256), 0, st, hdr, words));
    return SPEC_OK;
}

// Where the last level takes one warp per row.  A warp selects its lists 32 at a time, in as many rounds each time as a row has
// children (`rounds` in all), and a sequence's warps share an SM; the five warps of the other form have one to themselves while
// there are no more rows than SMs.  Draft of d 256 or 512, V 9000 to 128256, 1 to 256 sequences; us, this form less the other:
//   children  lists     one row a sequence;        2 to 24 rows; in all up to
//                       up to 48 / more sequences  48 rows        148 rows       592 rows       more
//   1, 2      36-148    -2.0..+0.1  -1.1..+1.0     -6.8..-1.4     -4.8..-0.6     -4.8..+1.4     -4.5..-0.2
//   4         36-148    -2.0..-0.2  -1.3..+3.2     -8.7..-0.2     -3.5..-0.2     -4.7..+1.2     -5.4..+1.9
//   8         71-148    -1.0..+1.5  +0.4..+9.2     -5.3..+2.8 *   -2.8..+5.6     -4.3..+2.9     -6.5..+8.9
//   1, 2, 4   223-255   --          --             --             -1.5..+2.3 *   -3.1..+1.2     -4.3..+0.1
//   8         223-255   --          --             --             +0.8..+7.9     -3.1..+4.8 *   -2.7..+1.1
//   1, 2      501-573   --          +1.4..+3.0     --             -0.3..+2.3     -1.4..+4.1     -2.6..+2.7
//   4, 8      501-573   --          +1.8..+7.2     --             +0.5..+26.2    -2.1..+19.9    +0.4..+13.1
// (* Most losses are those of sequences whose rows have more than 480 rounds together.)  Over these 1100 points and 228 of other
// branching factors (3 and 5 to 7 among them) the rule is 0.15 percent from the better form each time, the limits of 24 rows and
// 256 lists alone 0.5.
bool one_warp_per_row(const MergeArgs &g, int rows) {
    const int rounds = (g.n_tiles + 31) / 32 * g.topk;
    if (g.rows_per_seq > kPruneRows || g.n_tiles > 256) return false;
    if (g.rows_per_seq == 1) return rounds <= (rows <= 32 ? 35 : 15);
    if (rounds <= 24) return true;
    return (rows <= 48 || rows > num_sms()) && (g.rows_per_seq * rounds <= 480 || rows > 4 * num_sms());
}

int launch_merge_expand(const MergeArgs &g, int rows, cudaStream_t st) {
    const size_t smem = g.seq_done ? prune_smem_bytes(g.L, g.Lpad) : 0;
    const int slots = list_slots(g.list_len > 0 ? g.list_len : g.topk);
    if (g.seq_done && one_warp_per_row(g, rows)) {
        SPEC_CUDA_TRY(launch_pdl(slots == 2   ? merge_prune_kernel<2>
                                 : slots == 4 ? merge_prune_kernel<4>
                                              : merge_prune_kernel<8>, dim3(rows / g.rows_per_seq),
                                 dim3(32 * g.rows_per_seq), 0, st, g));
        return SPEC_OK;
    }
    SPEC_CUDA_TRY(launch_pdl(slots == 2   ? merge_expand_kernel<2>
                             : slots == 4 ? merge_expand_kernel<4>
                                          : merge_expand_kernel<8>, dim3(rows), dim3(kMergeThreads), smem, st, g));
    return SPEC_OK;
}

// Whether the LayerNorm sums of a level with `topk` children per row, behind a bf16 head, are taken in order (group_sums) in every
// kernel that may compute its states, so that these are the same bits whatever the number of rows.  In a tree, whose shape goes
// by the kernel and so by the number of rows, they are taken at the first level, behind three children and more or an e4m3 head,
// in a level that has an e4m3 copy, in rows of more than 4096 elements, of split vocabularies and with per-kernel profiling.
bool mix_sums_in_order(int topk, const MixArgs &m) {
    return topk <= kFusedChildren && m.S8_out == nullptr && m.d <= 8 * kRowThreads * 2;
}

// Returns SPEC_ERR_SHAPE when no fused form covers the shape (rows wider than 4096 elements; beyond one child per SM also other
// than two children per row, more rows than SMs, or an e4m3 copy of the states wanted): the caller then launches the merge and
// the mix separately.  More rows than SMs: the CTAs of a row with 512 threads take turns on the SMs, the separate kernels run in
// one wave.  384 rows of two children, d 4096: 22.9 us -> 18.0.
int launch_merge_mix(const MergeArgs &g, const MixArgs &m, int rows, cudaStream_t st) {
    if (m.d > 8 * kRowThreads * 2 || g.lse_out != nullptr || g.seq_done != nullptr) return SPEC_ERR_SHAPE;
    MergeMixArgs a{g, m};
    a.merge.next_emb = nullptr;   // the gather follows in the same CTA
    const int children = rows * g.topk, slots = list_slots(g.list_len > 0 ? g.list_len : g.topk);
    if (children <= num_sms()) {
        if (m.d > 8 * kRowThreads)
            SPEC_CUDA_TRY(launch_pdl(slots == 2   ? merge_mix_child_512_kernel<2>
                                     : slots == 4 ? merge_mix_child_512_kernel<4>
                                                  : merge_mix_child_512_kernel<8>, dim3(children),
                                     dim3(kWideRowThreads), 0, st, a));
        else
            SPEC_CUDA_TRY(launch_pdl(slots == 2   ? merge_mix_child_kernel<2>
                                     : slots == 4 ? merge_mix_child_kernel<4>
                                                  : merge_mix_child_kernel<8>, dim3(children),
                                     dim3(kRowThreads), 0, st, a));
        return SPEC_OK;
    }
    if (rows > num_sms() || g.topk != kFusedChildren || slots != list_slots(kFusedChildren) || m.S8_out != nullptr)
        return SPEC_ERR_SHAPE;
    if (m.d > 8 * kRowThreads) {
        SPEC_CUDA_TRY(launch_pdl(merge_mix_512_kernel, dim3(rows), dim3(kWideRowThreads), 0, st, a));
        return SPEC_OK;
    }
    SPEC_CUDA_TRY(launch_pdl(merge_mix_kernel, dim3(rows), dim3(kRowThreads), 0, st, a));
    return SPEC_OK;
}

int launch_merge_shards(const void *slots, size_t slot_bytes, int n_ranks, int rows, int topk, const float *score_in,
                        int32_t *tok_out, float *score_out, cudaStream_t st) {
    if (n_ranks < 1 || n_ranks > 32 || n_ranks * topk > 64) return SPEC_ERR_SHAPE;
    const int grid = (rows + kShardRowsPerCta - 1) / kShardRowsPerCta;
    SPEC_CUDA_TRY(launch_pdl(merge_shards_kernel, dim3(grid), dim3(32 * kShardRowsPerCta), 0, st, (const char *)slots,
                             slot_bytes, n_ranks, rows, topk, score_in, tok_out, score_out));
    return SPEC_OK;
}

int launch_prune(const float *leaf_score, const PruneArgs &pa, int B, int L, int K, int32_t *cand_tok,
                 float *cand_logp, cudaStream_t st) {
    int Lpad = 2;
    while (Lpad < L) Lpad <<= 1;
    SPEC_CUDA_TRY(launch_pdl(prune_kernel, dim3(B), dim3(kRowThreads), prune_smem_bytes(L, Lpad), st, leaf_score, pa,
                             L, Lpad, K, cand_tok, cand_logp));
    return SPEC_OK;
}

}  // namespace spec
