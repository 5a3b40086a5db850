// The whole draft of a small speculator in one kernel: one cluster of CTAs, the steps separated by cluster barriers
// instead of kernel boundaries.
//
// A draft of the smallest shapes reads a megabyte or two, and what it costs is its chain of 2 n + 2 dependent kernels
// (about 4.5 us each, and most of that again in host time).  Here the cluster's warps deal the rows of a level's matrices among
// themselves (16 rows per warp and item, mma.sync m16n8k16 with the weights read straight into fragments: there is no
// reuse of a weight that shared memory could serve), every CTA keeps all nodes of the level in its shared memory and
// repeats the merge and the mix of all of them, so that one barrier per level is enough: behind it every CTA has every
// CTA's partial lists (pushed through distributed shared memory) and the next level's projections (global memory).
//
//   P_0 | mix_0, P_1 + head_0 | merge_0, mix_1, P_2 + head_1 | ... | merge_last, prune      ("|": a cluster barrier)
//
// What bounds it: the latency of every step.  Per level of the smallest shape (V 1024, d 256, 1 / 4 / 12 nodes) mix 1.7 - 2.4,
// projection and head 1.0 - 1.2, selection 1.4 - 2.0, barrier 0.5, merge 0.9 us, the prune 0.9.  8 instead of 16 CTAs are
// 0.5 us faster there and 5 to 6 us slower at V 4096; 256 instead of 512 threads 2.5 us slower; requesting the level's weights
// into L1 before the mix gains nothing, nor do the arguments in shared memory; sums and lists of the selection in separate
// warps, which must then leave the logits as they are, cost it 2 us.  (Loads without predicates and the LayerNorm parameters,
// the tokens and the leaves in shared memory: 31.5 -> 28.2 us for the step.)
#include "row_ops.cuh"

namespace spec {

namespace {

using rows::float_key;
using rows::key_float;

constexpr int kCtas = 16;             // CTAs of the cluster
constexpr int kSmallThreads = 512;
constexpr int kSmallWarps = kSmallThreads / 32;
constexpr int kWarpsAll = kCtas * kSmallWarps;
constexpr int kMaxNodes = 16;        // nodes of a level whose head runs
constexpr int kMaxSplits = 4;        // K ranges of a projection
constexpr int kMaxSmem = 200 << 10;   // (16 nodes, V 4096, d_base 2048: 121 KB)

struct WarpSync {
    static __device__ __forceinline__ void sync() { __syncwarp(); }
};

struct SmallArgs {
    spec_weights_t w;
    const uint16_t *ctx;
    MixArgs mix[SPEC_MAX_HEADS];        // P: the level's own buffer of the two; p_splits as the projection was cut
    int32_t *tok[SPEC_MAX_HEADS + 1];
    float *score[SPEC_MAX_HEADS + 1];
    int32_t topk[SPEC_MAX_HEADS];
    int32_t *header;
    int header_words;
    int B, K, L;
    int32_t *cand_tok;
    float *cand_logp;
    int pitch_base, pitch;              // bytes between the rows of the operand in shared memory: 64 modulo 128
    int off_logits, logit_pitch;        // byte offset of the logits, floats between the nodes
    int off_lists, off_nodes, off_ln;   // byte offsets of the partial lists (two sets), the nodes, the LayerNorm parameters
};

// Partial list of one (node, CTA).
struct __align__(8) SmallList {
    float val[SPEC_MAX_TOPK];
    int id[SPEC_MAX_TOPK];
    float m, s;
};

__device__ __forceinline__ uint32_t small_rank() {
    uint32_t r;
    asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ void small_barrier() {
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

__device__ __forceinline__ uint4 ld_weights(const uint16_t *p, bool ok) {
    uint4 v = make_uint4(0u, 0u, 0u, 0u);
    if (ok) asm volatile("ld.global.nc.L1::no_allocate.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
    return v;
}

__device__ __forceinline__ void mma16816(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0,
                                         uint32_t b1) {
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
                 : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
                 : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

// Rows [row0, row0 + 16) of W [rows, Kd], elements [k0, k1) of each (multiples of 32 but for the last k1 = Kd), times the
// `nodes` operand rows in shared memory.  Lane (g, t) = (lane / 4, lane % 4) holds the elements 8 t .. 8 t + 7 of a group of
// 32 of rows g and g + 8 and of node g: one 16-byte load each, two MMAs.  (The order of k inside a group is the same
// permutation on both sides.)  c[q]: nodes 8 q + 2 t, + 1 of row g, then of row g + 8.
constexpr int kGroups = kMaxNodes / 8;
constexpr int kAhead = 8;   // groups of 32 elements whose loads are in flight together
__device__ __forceinline__ void tile_times_nodes(const uint16_t *W, int rows, int Kd, int row0, int k0, int k1,
                                                 const char *x, int pitch, int nodes, int lane, float (&c)[kGroups][4]) {
    const int g = lane >> 2, t = lane & 3;
#pragma unroll
    for (int q = 0; q < kGroups; ++q) c[q][0] = c[q][1] = c[q][2] = c[q][3] = 0.0f;
    // (a row past the last one is read as the first: its results go nowhere)
    const uint16_t *w0 = W + (size_t)(row0 + g < rows ? row0 + g : 0) * Kd + k0 + 8 * t;
    const uint16_t *w1 = W + (size_t)(row0 + g + 8 < rows ? row0 + g + 8 : 0) * Kd + k0 + 8 * t;
    const char *xg = x + g * pitch + 2 * k0 + 16 * t;
    const bool second = nodes > 8;
    auto multiply = [&](const uint4 &p, const uint4 &q, const char *at) {
        // (rows past the last node hold something finite and their results go nowhere either)
        const uint4 b = *(const uint4 *)at;
        mma16816(c[0], p.x, q.x, p.y, q.y, b.x, b.y);
        mma16816(c[0], p.z, q.z, p.w, q.w, b.z, b.w);
        if (second) {
            const uint4 e = *(const uint4 *)(at + 8 * pitch);
            mma16816(c[1], p.x, q.x, p.y, q.y, e.x, e.y);
            mma16816(c[1], p.z, q.z, p.w, q.w, e.z, e.w);
        }
    };
    static_assert(kGroups == 2, "multiply");
    int left = k1 - k0;
    for (; left >= 32 * kAhead; left -= 32 * kAhead) {
        uint4 a0[kAhead], a1[kAhead];
#pragma unroll
        for (int u = 0; u < kAhead; ++u) {
            a0[u] = ld_weights(w0 + 32 * u, true);
            a1[u] = ld_weights(w1 + 32 * u, true);
        }
#pragma unroll
        for (int u = 0; u < kAhead; ++u) multiply(a0[u], a1[u], xg + 64 * u);
        w0 += 32 * kAhead;
        w1 += 32 * kAhead;
        xg += 64 * kAhead;
    }
    if (left > 0) {
        uint4 a0[kAhead], a1[kAhead];
#pragma unroll
        for (int u = 0; u < kAhead; ++u) {
            const bool in = 32 * u + 8 * t < left;
            a0[u] = ld_weights(w0 + 32 * u, in);
            a1[u] = ld_weights(w1 + 32 * u, in);
        }
#pragma unroll
        for (int u = 0; u < kAhead; ++u) {
            if (32 * u >= left) break;   // (uniform)
            multiply(a0[u], a1[u], xg + 64 * u);
        }
    }
}

// One item of the projection W [d, Kd] of `nodes` parents: item i = (split, tile).  P [split][nodes][d].
__device__ __forceinline__ void project(const uint16_t *W, int d, int Kd, int splits, int item, const char *x, int pitch,
                                        int nodes, float *P, size_t split_stride, int lane) {
    const int tiles = (d + 15) / 16, split = item / tiles, row0 = (item - split * tiles) * 16;
    const int per = ((Kd + 31) / 32 + splits - 1) / splits * 32, k0 = split * per, k1 = min(Kd, k0 + per);
    float c[kGroups][4];
    tile_times_nodes(W, d, Kd, row0, k0, k1, x, pitch, nodes, lane, c);
    const int r = row0 + (lane >> 2), n0 = 2 * (lane & 3);
    float *out = P + split * split_stride + (n0 * d + r);
#pragma unroll
    for (int q = 0; q < kGroups; ++q) {
        if (8 * q >= nodes) break;
        const bool n_ok = 8 * q + n0 < nodes, n1_ok = 8 * q + n0 + 1 < nodes;
        float *o = out + 8 * q * d;
        if (n_ok && r < d) o[0] = c[q][0];
        if (n1_ok && r < d) o[d] = c[q][1];
        if (n_ok && r + 8 < d) o[8] = c[q][2];
        if (n1_ok && r + 8 < d) o[d + 8] = c[q][3];
    }
}

__global__ void __launch_bounds__(kSmallThreads, 1) draft_small_kernel(const __grid_constant__ SmallArgs a) {
    extern __shared__ __align__(128) char smem[];
    __shared__ float red[kSmallWarps][2 * rows::kMaxGroupWarps];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, rank = (int)small_rank();
    const int gw = warp * kCtas + rank;   // item i belongs to warp i % kWarpsAll: to CTA i % kCtas
    const int d = a.w.d_inner, V = a.w.V, n = a.w.n_heads;
    char *x = smem;
    float *logits = (float *)(smem + a.off_logits);
    SmallList *lists = (SmallList *)(smem + a.off_lists);           // [2][kMaxNodes][kCtas]
    constexpr int kLevel = kMaxNodes * SPEC_MAX_TOPK;               // most nodes of a level
    int *node_tok = (int *)(smem + a.off_nodes);                    // [n + 1][kLevel]: the nodes' tokens, every level's ...
    float *node_score = (float *)(node_tok + (n + 1) * kLevel);     // ... their scores, two sets by turns
    griddep_launch();
    float *ln = (float *)(smem + a.off_ln);   // [n][2][d]: the LayerNorm parameters
    for (int i = tid * 16; i < a.off_logits; i += kSmallThreads * 16) *(uint4 *)(smem + i) = make_uint4(0u, 0u, 0u, 0u);
    __syncthreads();
    griddep_wait();
    if (rank == 0)
        for (int i = tid; i < a.header_words; i += kSmallThreads) a.header[i] = 0;
    // the context states
    const int base_vec = a.w.d_base / 8;
    for (int i = tid; i < a.B * base_vec; i += kSmallThreads) {
        const int b = i / base_vec, v = i - b * base_vec;
        *(uint4 *)(x + b * a.pitch_base + 16 * v) = __ldcg((const uint4 *)a.ctx + i);
    }
    for (int b = tid; b < a.B; b += kSmallThreads) node_tok[b] = __ldcg(a.mix[0].tok + b);
    __syncthreads();
    const int tiles_d = (d + 15) / 16, tiles_v = (V + 15) / 16;
    for (int i = gw; i < tiles_d * a.mix[0].p_splits; i += kWarpsAll)
        project((const uint16_t *)a.w.proj[0], d, a.w.d_base, a.mix[0].p_splits, i, x, a.pitch_base, a.B, (float *)a.mix[0].P,
                a.mix[0].p_split_stride, lane);
    // The LayerNorm parameters, like everything else not before the wait: a kernel earlier in the stream may have written them.
    // Loaded by the warps that the projection leaves idle (32 tiles times four splits are half of the cluster's warps) and only
    // behind its code: ahead of it, or by all warps, the smallest step took 0.4 us longer.
    if (warp >= kSmallWarps / 2) {
        const int u = tid - kSmallThreads / 2;
#pragma unroll 1
        for (int i = u; i < n * d / 2; i += kSmallThreads / 2) {
            const int l = i / (d / 2), j = 4 * (i - l * (d / 2));
            *(float4 *)(ln + l * 2 * d + j) = __ldcg((const float4 *)(j < d ? a.w.ln_gamma[l] + j : a.w.ln_beta[l] + (j - d)));
        }
    }
    small_barrier();   // (also: every CTA of the cluster runs, its shared memory may be written)

    int nodes = a.B;
    for (int l = 0; l < n; ++l) {
        // the states of the level's nodes, all of them in every CTA
        MixArgs m = a.mix[l];
        const int parent_div = m.parent_div;
        if (l == 0) {   // (the pad of the rows below held context states)
            for (int i = tid * 16; i < kMaxNodes * a.pitch; i += kSmallThreads * 16) *(uint4 *)(x + i) = make_uint4(0u, 0u, 0u, 0u);
            __syncthreads();
        }
        uint16_t *S = m.S_out;
        for (int i = warp; i < nodes; i += kSmallWarps) {
            m.S_out = (uint16_t *)(x + i * a.pitch);
            m.gamma = ln + l * 2 * d;
            m.beta = m.gamma + d;
            m.err = rank == 0 ? a.mix[l].err : nullptr;
            if (d <= 256) rows::mix_ln_gelu_row<32, 1, 1, WarpSync, kMaxSplits>(m, 0, i / parent_div, node_tok[l * kLevel + i], lane, red[warp]);
            else rows::mix_ln_gelu_row<32, 2, 1, WarpSync, kMaxSplits>(m, 0, i / parent_div, node_tok[l * kLevel + i], lane, red[warp]);
        }
        __syncthreads();
        // the next level's projection and this level's head
        const int splits = l + 1 < n ? a.mix[l + 1].p_splits : 0, n_proj = tiles_d * splits;
        const int head_rank = (rank + kCtas - n_proj % kCtas) % kCtas;   // head tile h is this CTA's if h % kCtas is this
        for (int i = gw; i < n_proj + tiles_v; i += kWarpsAll) {
            if (i < n_proj) {
                project((const uint16_t *)a.w.proj[l + 1], d, d, splits, i, x, a.pitch, nodes, (float *)a.mix[l + 1].P,
                        a.mix[l + 1].p_split_stride, lane);
            } else {
                const int tile = i - n_proj, row0 = 16 * tile, col0 = 16 * (tile / kCtas);
                float c[kGroups][4];
                tile_times_nodes((const uint16_t *)a.w.head[l], V, d, row0, 0, d, x, a.pitch, nodes, lane, c);
                const int r = lane >> 2, pitch = a.logit_pitch;
                const bool v0 = row0 + r < V, v1 = row0 + r + 8 < V;
                float *out = logits + 2 * (lane & 3) * pitch + col0 + r;   // (rows of the nodes rounded up to eight are there)
#pragma unroll
                for (int q = 0; q < kGroups; ++q) {
                    if (8 * q >= nodes) break;
                    float *o = out + 8 * q * pitch;
                    o[0] = v0 ? c[q][0] : -INFINITY;
                    o[pitch] = v0 ? c[q][1] : -INFINITY;
                    o[8] = v1 ? c[q][2] : -INFINITY;
                    o[pitch + 8] = v1 ? c[q][3] : -INFINITY;
                }
            }
        }
        if (rank == 0)   // for the caller's eyes (spec_draft_layout)
            for (int i = tid; i < nodes * (d / 8); i += kSmallThreads) {
                const int r = i / (d / 8), v = i - r * (d / 8);
                *((uint4 *)S + i) = *(const uint4 *)(x + r * a.pitch + 16 * v);
            }
        __syncthreads();
        // this CTA's partial list of every node, to every CTA
        const int topk = a.topk[l];
        const int cols = 16 * ((tiles_v - head_rank + kCtas - 1) / kCtas);
        SmallList *set = lists + (l & 1) * kMaxNodes * kCtas;
        for (int i = warp; i < nodes; i += kSmallWarps) {
            float *row = logits + i * a.logit_pitch;
            // the lane's two best entries that are left, the lowest id first among equals
            float v, v2;
            int col, col2;
            auto scan = [&]() {
                v = v2 = -INFINITY;
                col = col2 = -1;
#pragma unroll 4
                for (int j = lane; j < cols; j += 32) {
                    const float y = row[j];
                    const bool first = y > v, second = y > v2;
                    v2 = first ? v : (second ? y : v2);
                    col2 = first ? col : (second ? j : col2);
                    v = first ? y : v;
                    col = first ? j : col;
                }
            };
            auto id_of = [&](int col) { return col < 0 ? 0x7fffffff : ((col >> 4) * kCtas + head_rank) * 16 + (col & 15); };
            scan();
            const float mx = key_float(__reduce_max_sync(0xffffffffu, float_key(v)));
            float s = 0.0f;
            if (mx > -INFINITY) {
#pragma unroll 4
                for (int j = lane; j < cols; j += 32) s += __expf(row[j] - mx);
            }
#pragma unroll
            for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
            float lv = -INFINITY;
            int li = 0x7fffffff;
            for (int j = 0; j < topk; ++j) {
                const uint32_t key = float_key(v);
                const uint32_t bk = __reduce_max_sync(0xffffffffu, key);
                const int id = id_of(col);
                const int bi = (int)__reduce_min_sync(0xffffffffu, key == bk ? (uint32_t)id : 0xffffffffu);
                if (lane == j) {
                    lv = key_float(bk);
                    li = bi;
                }
                if (key == bk && id == bi && col >= 0) {
                    row[col] = -INFINITY;
                    v = v2;
                    col = col2;
                    v2 = -INFINITY;
                    if (col2 < 0) scan();   // both gone
                    col2 = -1;
                }
            }
            SmallList *mine = set + i * kCtas + rank;
#pragma unroll
            for (int q = 0; q < kCtas; ++q) {
                if (lane < topk || lane == 31) {
                    const uint32_t at = (uint32_t)__cvta_generic_to_shared(lane == 31 ? (void *)&mine->m : (void *)&mine->val[lane]);
                    uint32_t there;
                    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(there) : "r"(at), "r"(q));
                    const uint32_t first = __float_as_uint(lane == 31 ? mx : lv), second = lane == 31 ? __float_as_uint(s) : (uint32_t)li;
                    const int step = lane == 31 ? 4 : (int)sizeof(float) * SPEC_MAX_TOPK;
                    asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(there), "r"(first) : "memory");
                    asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(there + step), "r"(second) : "memory");
                }
            }
        }
        small_barrier();
        // the nodes' children, in every CTA
        const float *score_in = node_score + (l & 1) * kLevel;
        float *score_out = node_score + ((l + 1) & 1) * kLevel;
        for (int i = warp; i < nodes; i += kSmallWarps) {
            const SmallList *li = set + i * kCtas + (lane < kCtas ? lane : 0);
            const float pm = lane < kCtas ? li->m : -INFINITY, ps = lane < kCtas ? li->s : 0.0f;
            float mx = pm;
#pragma unroll
            for (int off = 16; off > 0; off >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, off));
            float s = pm > -INFINITY ? ps * __expf(pm - mx) : 0.0f;
#pragma unroll
            for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
            const float lse = mx + logf(s), base = l == 0 ? 0.0f : score_in[i];
            int used = 0;
            uint32_t hk = float_key(lane < kCtas ? li->val[0] : -INFINITY);
            int hi = lane < kCtas ? li->id[0] : 0x7fffffff;
            for (int j = 0; j < topk; ++j) {
                const uint32_t bk = __reduce_max_sync(0xffffffffu, hk);
                const int bi = (int)__reduce_min_sync(0xffffffffu, hk == bk ? (uint32_t)hi : 0xffffffffu);
                if (lane == 0) {
                    const int child = i * topk + j;
                    const float score = base + (key_float(bk) - lse);
                    node_tok[(l + 1) * kLevel + child] = bi;
                    score_out[child] = score;
                    if (rank == 0) {
                        a.tok[l + 1][child] = bi;
                        a.score[l + 1][child] = score;
                    }
                }
                if (hk == bk && hi == bi && lane < kCtas) {
                    ++used;
                    hk = float_key(used < topk ? li->val[used] : -INFINITY);
                    hi = used < topk ? li->id[used] : 0x7fffffff;
                }
            }
        }
        __syncthreads();
        nodes *= topk;
    }
    // the K best leaves of every sequence by (score desc, leaf asc): a thread's rank is the leaves that precede its own
    if (rank == 0 && tid < nodes) {
        const float *score = node_score + (n & 1) * kLevel;
        const int b = tid / a.L, leaf = tid - b * a.L;
        const rows::LeafKey mine = {score[tid], leaf};
        int before = 0;
        for (int j = 0; j < a.L; ++j) before += rows::leaf_before({score[b * a.L + j], j}, mine) ? 1 : 0;
        if (before < a.K) {
            const size_t out = (size_t)b * a.K + before;
            a.cand_logp[out] = mine.score;
            int idx = tid;
            for (int l = n; l > 0; --l) {
                a.cand_tok[out * n + l - 1] = node_tok[l * kLevel + idx];
                idx /= a.topk[l - 1];
            }
        }
    }
}

int pitch_of(int elems) { return (2 * elems + 127) / 128 * 128 + 64; }

}  // namespace

// Which drafts run as one kernel: those whose levels read little for the sixteen CTAs (a megabyte each way costs 2 to 3 us,
// in the kernel chain a fifth of that), the less the more nodes every CTA has to mix and to select for.  us per draft, kernel
// chain -> one kernel, d_base 512, branching 4, 3, 2 unless stated: V 1000, d 256 39.7 -> 23; V 4096, d 256 39.5 -> 27.0;
// V 5400, d 256 40.4 -> 30.3; V 2000, d 512 41.5 -> 30.4; V 2700, d 512 41.6 -> 33.2; branching 6, 2 for two sequences, V 1500,
// d 504 31.6 -> 22.5; one level, V 1200, d 256 16.8 -> 9.7; chains of three for 16 sequences, V 1000, d 256 38.0 -> 26.2,
// V 3600, d 256 38.1 -> 31.8, V 1800, d 512 39.6 -> 38.2; a chain of five for one, V 3400, d 512 61.1 -> 50.1.  Far beyond
// the line (3 us more per draft then): V 6000, d 512 42.6 -> 52.7; V 16000, d 256 41.1 -> 56.3; 32 nodes, with room for
// them, V 2000, d 256 40.8 -> 47.4.  The smallest decoding step 45.7 -> 28.2.
bool small_draft_fits(const spec_weights_t &w, int B, const int32_t *topk) {
    if (w.d_inner > 512 || w.d_base > 2048) return false;
    long long nodes = B, cost = 0;
    for (int l = 0; l < w.n_heads; ++l) {
        if (nodes > kMaxNodes) return false;
        cost += (long long)w.V * w.d_inner * (16 + nodes);
        nodes *= topk[l];
    }
    return cost <= (30ll << 20) * w.n_heads;
}

// Floats of the two projection buffers together.
size_t small_draft_proj_floats(const spec_weights_t &w) { return (size_t)2 * kMaxSplits * kMaxNodes * w.d_inner; }

int launch_draft_small(const spec_weights_t &w, const void *ctx, int B, const int32_t *topk, int K, const MixArgs *mix,
                       int32_t *const *tok, float *const *score, float *proj, int32_t *header, int header_words,
                       int L, int32_t *cand_tok, float *cand_logp, cudaStream_t st) {
    SmallArgs a{};
    a.w = w;
    a.ctx = (const uint16_t *)ctx;
    const int n = w.n_heads, tiles_d = (w.d_inner + 15) / 16;
    int parents = B, max_nodes = B;
    for (int l = 0; l < n; ++l) {
        const int groups = ((l == 0 ? w.d_base : w.d_inner) + 31) / 32;
        int splits = kWarpsAll / tiles_d;   // no warp with a second item
        if (splits > kMaxSplits) splits = kMaxSplits;
        if (splits > (groups + 1) / 2) splits = (groups + 1) / 2;
        if (splits < 1) splits = 1;
        const int per = (groups + splits - 1) / splits;
        splits = (groups + per - 1) / per;   // no empty range
        a.mix[l] = mix[l];
        a.mix[l].P = proj + (size_t)(l & 1) * kMaxSplits * kMaxNodes * w.d_inner;
        a.mix[l].p_splits = splits;
        a.mix[l].p_split_stride = (size_t)parents * w.d_inner;
        parents = l == 0 ? B : parents * topk[l - 1];
        if (parents > max_nodes) max_nodes = parents;
        a.topk[l] = topk[l];
    }
    for (int l = 1; l <= n; ++l) {
        a.tok[l] = tok[l];
        a.score[l] = score[l];
    }
    a.header = header;
    a.header_words = header_words;
    a.B = B; a.K = K; a.L = L;
    a.cand_tok = cand_tok;
    a.cand_logp = cand_logp;
    a.pitch_base = pitch_of(w.d_base);
    a.pitch = pitch_of(w.d_inner);
    const int node_rows = (max_nodes + 7) / 8 * 8;
    const int base_rows = (B + 7) / 8 * 8;
    int off = kMaxNodes * a.pitch;
    if (base_rows * a.pitch_base > off) off = base_rows * a.pitch_base;
    a.off_logits = (off + 127) / 128 * 128;
    a.logit_pitch = 16 * (((w.V + 15) / 16 + kCtas - 1) / kCtas) + 1;
    off = a.off_logits + 4 * node_rows * a.logit_pitch;
    a.off_lists = (off + 127) / 128 * 128;
    off = a.off_lists + 2 * kMaxNodes * kCtas * (int)sizeof(SmallList);
    a.off_nodes = (off + 127) / 128 * 128;
    off = a.off_nodes + (n + 3) * 4 * kMaxNodes * SPEC_MAX_TOPK;
    a.off_ln = (off + 127) / 128 * 128;
    off = a.off_ln + n * 2 * 4 * w.d_inner;
    if (off > kMaxSmem) return SPEC_ERR_SHAPE;
    // Asked for on every call (0.3 us), for the stream and the context that it is made in: another one may have fewer SMs.
    SPEC_CUDA_TRY(cudaFuncSetAttribute(draft_small_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxSmem));
    SPEC_CUDA_TRY(cudaFuncSetAttribute(draft_small_kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(kCtas);
    cfg.blockDim = dim3(kSmallThreads);
    cfg.dynamicSmemBytes = (size_t)off;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = kCtas;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int fit = 0;
    if (cudaOccupancyMaxActiveClusters(&fit, draft_small_kernel, &cfg) != cudaSuccess || fit < 1) {
        (void)cudaGetLastError();
        return SPEC_ERR_SHAPE;   // fewer SMs side by side than a cluster wants
    }
    SPEC_CUDA_TRY(launch_pdl_cluster(draft_small_kernel, dim3(kCtas), dim3(kSmallThreads), (size_t)off, kCtas, st, a));
    return SPEC_OK;
}

}  // namespace spec
