// Row-wise steps of the draft path (Sec. 3.1 / Sec. 4.1 of arXiv 2404.19124), written for a group of
// kThreads threads that synchronises through `Sync::sync()` (a whole CTA in the stand-alone kernels).
//   mix_ln_gelu_row   embedding gather + weighted mix with the projected parent state (sum of the
//                     split-K partials) + LayerNorm + exact GELU for one tree node, bf16 state out
//   merge_expand_row  folds the per-tile partial top-k lists and (max, sum-exp) pairs of one row into
//                     its top-k tokens and log-probabilities and writes the node's children
//   prune_sequence    orders one sequence's leaves by (score desc, leaf index asc), keeps K, walks
//                     back to the root to emit the K n-grams
// These steps run once per launch on a handful of rows, so what they cost is latency: every load of a
// step is issued before the first one is used, and dependent chains are kept short.
// Buffers that a preceding kernel wrote are read with ld.global.cg, never through the non-coherent path.
#pragma once

#include <math.h>

#include "fp8.cuh"
#include "spec_common.cuh"

namespace spec {
namespace rows {

using spec::MergeArgs;
using spec::MixArgs;

struct BlockSync {
    static __device__ __forceinline__ void sync() { __syncthreads(); }
};

// Scratch in shared memory for one group.
constexpr int kMaxGroupWarps = 16;
constexpr int kMaxRounds = 16;        // most entries a selection can return (top-k itself needs at most 8)
struct Scratch {
    float red_m[kMaxGroupWarps], red_s[kMaxGroupWarps];
    uint32_t cand_k[kMaxGroupWarps][kMaxRounds];   // every warp's best entries, best first: value keys ...
    int cand_i[kMaxGroupWarps][kMaxRounds];        // ... and token ids
};

// (`red`: one float per warp, not read by anybody else until the next barrier behind the call.)
template <int kThreads, typename Sync>   // (kThreads 0: blockDim.x)
__device__ __forceinline__ float group_sum(float v, float *red, int tid) {
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
    if (kThreads == 32) return v;
    const int w = tid >> 5, l = tid & 31;
    if (l == 0) red[w] = v;
    Sync::sync();
    const int warps = (kThreads > 0 ? kThreads : (int)blockDim.x) / 32;
    float t = l < warps ? red[l] : 0.0f;
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) t += __shfl_xor_sync(0xffffffffu, t, off);
    return t;
}

// The sum over a row of which a thread holds kIters groups of eight.  `in_order`: v[it] is the sum of group it, 256 elements are
// summed at a time and those sums added one after the other, as mix_children adds them; else v[kIters - 1] is the sum of all
// of the thread's groups, and the threads' are added in a tree.
template <int kThreads, int kIters, typename Sync>
__device__ __forceinline__ float group_sums(const float (&v)[kIters], float *red, int tid, bool in_order) {
    if (in_order) {   // (uniform)
        const int warps = (kThreads > 0 ? kThreads : (int)blockDim.x) / 32;
#pragma unroll
        for (int it = 0; it < kIters; ++it) {
            float x = v[it];
#pragma unroll
            for (int off = 16; off > 0; off >>= 1) x += __shfl_xor_sync(0xffffffffu, x, off);
            if ((tid & 31) == 0) red[it * warps + (tid >> 5)] = x;
        }
        Sync::sync();
        float t = 0.0f;
#pragma unroll
        for (int q = 0; q < kIters * warps; ++q) t += red[q];
        return t;
    }
    return group_sum<kThreads, Sync>(v[kIters - 1], red, tid);
}

template <int kThreads, typename Sync>
__device__ __forceinline__ float group_max(float v, float *red, int tid) {
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, off));
    const int w = tid >> 5, l = tid & 31;
    Sync::sync();
    if (l == 0) red[w] = v;
    Sync::sync();
    float t = l < (kThreads > 0 ? kThreads : (int)blockDim.x) / 32 ? red[l] : 0.0f;   // used for magnitudes only
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) t = fmaxf(t, __shfl_xor_sync(0xffffffffu, t, off));
    return t;
}

// Exact (erf) GELU.  erff is kept out of line: inlined it would be the bulk of the row step's code.  Four at a time, whose
// latency chains overlap (one by one the eight evaluations of a thread were a third of the step).
__device__ __forceinline__ float gelu_erf(float y) { return 0.5f * y * (1.0f + erff(y * 0.70710678118654752440f)); }
static __device__ __noinline__ float4 gelu_erf4(float4 y) {
    return make_float4(gelu_erf(y.x), gelu_erf(y.y), gelu_erf(y.z), gelu_erf(y.w));
}

// An element of the mixed row.  Which of the two products is rounded before the sum is spelt out: left to the compiler it
// differed from one kernel to the next, and with it, now and then, the bf16 value that a state is rounded to.
__device__ __forceinline__ float mix_element(const MixArgs &m, float p, float z) { return fmaf(m.b, z, __fmul_rn(m.a, p)); }

// Eight floats of a projection, 32-byte aligned (rows are whole groups of eight in the workspace), in one load.  Two 16-byte
// loads of a warp would each touch every 32-byte sector of the kilobyte and use half of it.
struct Float8 {
    float v[8];
};
__device__ __forceinline__ Float8 ldcg8(const float *p) {
    Float8 r;
    asm volatile("ld.global.cg.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=f"(r.v[0]), "=f"(r.v[1]), "=f"(r.v[2]), "=f"(r.v[3]), "=f"(r.v[4]), "=f"(r.v[5]), "=f"(r.v[6]), "=f"(r.v[7])
                 : "l"(p));
    return r;
}

// The projected parent state (the sum of its partials, added in ascending order) of the groups that thread `tid` owns in
// mix_ln_gelu_row with one group per thread.
template <int kThreads>
__device__ __forceinline__ void parent_state(const MixArgs &m, int parent, int tid, float (&pre)[1][8]) {
    const int i = tid * 8;
#pragma unroll
    for (int j = 0; j < 8; ++j) pre[0][j] = 0.0f;
    if (i >= m.d) return;
    const float *p = m.P + (size_t)parent * m.d + i;
    for (int s0 = 0; s0 < m.p_splits; s0 += 4) {
        Float8 a[4];
#pragma unroll
        for (int sp = 0; sp < 4; ++sp) {
            a[sp] = Float8{};
            if (s0 + sp < m.p_splits) a[sp] = ldcg8(p + (s0 + sp) * m.p_split_stride);
        }
#pragma unroll
        for (int sp = 0; sp < 4; ++sp) {
#pragma unroll
            for (int j = 0; j < 8; ++j) pre[0][j] += a[sp].v[j];
        }
    }
}

// Node r of the level, whose token is t and whose projected parent state is row `parent` of P.
// h = a * P[parent] + b * E[t].  The row lives in registers: thread t owns the 8-element groups
// t, t + kThreads, ... (kIters of them; d <= 8 * kThreads * kIters, d % 8 == 0; kThreads 0: as many as the CTA has).
// kDepth of those groups, and kSp partial projections of each, have their loads in flight together (registers against
// latency).
// `pre`: the projected parent state of this thread's groups (parent_state), if the caller has it already.  `in_order`: see
// group_sums (at most two groups).
template <int kThreads, int kIters, int kDepth, typename Sync, int kSp = 4>
__device__ __forceinline__ void mix_ln_gelu_row(const MixArgs &m, int r, int parent, int t, int tid, float *red,
                                                const float (*pre)[8] = nullptr, bool in_order = false) {
    constexpr int kGroup = kIters >= 8 ? 1 : (kIters < kDepth ? kIters : kDepth);
    bool tok_ok = false;
    const int nt = kThreads > 0 ? kThreads : (int)blockDim.x;
    const int d = m.d;
    const float *p = m.P + (size_t)parent * d;
    const uint16_t *e = nullptr;

    float h[kIters][8];
    float sums[kIters];
    const bool ordered = kIters <= 2 && in_order;
#pragma unroll
    for (int g0 = 0; g0 < kIters; g0 += kGroup) {
        // every load of the group is issued before the first value is used: one round trip per group
        uint4 ev[kGroup];
        Float8 pa[kGroup][kSp];
#pragma unroll
        for (int q = 0; q < kGroup; ++q) {
            const int i = ((g0 + q) * nt + tid) * 8;
#pragma unroll
            for (int sp = 0; sp < kSp; ++sp) {
                pa[q][sp] = Float8{};
                if (pre == nullptr && i < d && sp < m.p_splits) pa[q][sp] = ldcg8(p + sp * m.p_split_stride + i);
            }
        }
        if (g0 == 0) {   // (only now: everything above is in flight while the token arrives)
            tok_ok = (t >= 0) && (t < m.V);
            if (!tok_ok && tid == 0) report_error(m.err, SPEC_ERR_TOKEN_RANGE);
            e = m.emb + (size_t)(tok_ok ? t : 0) * d;
        }
#pragma unroll
        for (int q = 0; q < kGroup; ++q) {
            const int i = ((g0 + q) * nt + tid) * 8;
            ev[q] = make_uint4(0u, 0u, 0u, 0u);
            if (i < d && tok_ok) ev[q] = *(const uint4 *)(e + i);
        }
#pragma unroll
        for (int q = 0; q < kGroup; ++q) {
            const int it = g0 + q;
            const int i = (it * nt + tid) * 8;
            float pv[8] = {0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll
            for (int sp = 0; sp < kSp; ++sp) {      // partials are added in ascending order: reproducible
#pragma unroll
                for (int j = 0; j < 8; ++j) pv[j] += pa[q][sp].v[j];
            }
            if (pre != nullptr) {
#pragma unroll
                for (int j = 0; j < 8; ++j) pv[j] = pre[it][j];
            } else if (i < d) {
                for (int sp = kSp; sp < m.p_splits; ++sp) {   // more partials than one batch holds (rare)
                    const Float8 x = ldcg8(p + sp * m.p_split_stride + i);
#pragma unroll
                    for (int j = 0; j < 8; ++j) pv[j] += x.v[j];
                }
            }
            const uint32_t ew[4] = {ev[q].x, ev[q].y, ev[q].z, ev[q].w};
            float sum = it > 0 && !ordered ? sums[it > 0 ? it - 1 : 0] : 0.0f;
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const float z = (j & 1) ? __uint_as_float(ew[j >> 1] & 0xffff0000u) : __uint_as_float(ew[j >> 1] << 16);
                h[it][j] = i < d ? mix_element(m, pv[j], z) : 0.0f;
                sum += h[it][j];
            }
            sums[it] = sum;
        }
    }
    // LayerNorm parameters: requested before the two reductions so that they arrive while those run
    // (for the widest rows they are fetched where they are used, to stay within the register file)
    constexpr bool kHoist = kIters <= 2;
    constexpr int kHeld = kHoist ? kIters : 1;
    float4 gq[kHeld][2], bq[kHeld][2];
    if (kHoist) {
#pragma unroll
        for (int it = 0; it < kHeld; ++it) {
            const int i = (it * nt + tid) * 8;
            const int ic = i < d ? i : 0;
            gq[it][0] = *(const float4 *)(m.gamma + ic);
            gq[it][1] = *(const float4 *)(m.gamma + ic + 4);
            bq[it][0] = *(const float4 *)(m.beta + ic);
            bq[it][1] = *(const float4 *)(m.beta + ic + 4);
        }
    }
    const float mean = group_sums<kThreads, kIters, Sync>(sums, red, tid, ordered) / (float)d;
#pragma unroll
    for (int it = 0; it < kIters; ++it) {
        const int i = (it * nt + tid) * 8;
        float sq = it > 0 && !ordered ? sums[it > 0 ? it - 1 : 0] : 0.0f;
        if (i < d) {
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const float c = h[it][j] - mean;
                sq += c * c;
            }
        }
        sums[it] = sq;
    }
    const float var = group_sums<kThreads, kIters, Sync>(sums, red + kMaxGroupWarps, tid, ordered) / (float)d;
    const float rstd = rsqrtf(var + m.eps);
    float amax = 0.0f;   // largest magnitude of the bf16-rounded state (for the e4m3 copy); h is reused for it
#pragma unroll
    for (int it = 0; it < kIters; ++it) {
        const int i = (it * nt + tid) * 8;
        const int hq = kHoist ? it : 0;
        if (!kHoist) {
            const int ic = i < d ? i : 0;
            gq[0][0] = *(const float4 *)(m.gamma + ic);
            gq[0][1] = *(const float4 *)(m.gamma + ic + 4);
            bq[0][0] = *(const float4 *)(m.beta + ic);
            bq[0][1] = *(const float4 *)(m.beta + ic + 4);
        }
        const float gv[8] = {gq[hq][0].x, gq[hq][0].y, gq[hq][0].z, gq[hq][0].w, gq[hq][1].x, gq[hq][1].y, gq[hq][1].z, gq[hq][1].w};
        const float bv[8] = {bq[hq][0].x, bq[hq][0].y, bq[hq][0].z, bq[hq][0].w, bq[hq][1].x, bq[hq][1].y, bq[hq][1].z, bq[hq][1].w};
        uint32_t packed[4];
#pragma unroll
        for (int j = 0; j < 8; j += 4) {
            float4 y;
            y.x = (h[it][j] - mean) * rstd * gv[j] + bv[j];
            y.y = (h[it][j + 1] - mean) * rstd * gv[j + 1] + bv[j + 1];
            y.z = (h[it][j + 2] - mean) * rstd * gv[j + 2] + bv[j + 2];
            y.w = (h[it][j + 3] - mean) * rstd * gv[j + 3] + bv[j + 3];
            y = gelu_erf4(y);
            packed[j >> 1] = pack_bf16x2(y.x, y.y);
            packed[(j >> 1) + 1] = pack_bf16x2(y.z, y.w);
        }
        if (m.S8_out != nullptr) {   // (uniform)
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const uint32_t w = packed[j >> 1];
                h[it][j] = i < d ? __uint_as_float((j & 1) ? w & 0xffff0000u : w << 16) : 0.0f;
                amax = fmaxf(amax, fabsf(h[it][j]));
            }
        }
        if (i < d) *(uint4 *)(m.S_out + (size_t)r * d + i) = make_uint4(packed[0], packed[1], packed[2], packed[3]);
    }
    if (m.S8_out != nullptr) {   // uniform over the group
        const float scale = row_scale_of(group_max<kThreads, Sync>(amax, red, tid));
        const float inv = 1.0f / scale;
#pragma unroll
        for (int it = 0; it < kIters; ++it) {
            const int i = (it * nt + tid) * 8;
            if (i < d) *(uint2 *)(m.S8_out + (size_t)r * d + i) = e4m3x8(h[it], inv);
        }
        if (tid == 0) m.s8_scale[r] = scale;
    }
}

// (value desc, token id asc) ordering of candidates.
// Written without short-circuit operators and the exchanges below as selects: with "||" / "&&" and an "if"
// around the swap every comparison became a data-dependent branch that diverges inside the warp, and one
// 8-entry list took 2000-6000 cycles to fold instead of a few hundred.
__device__ __forceinline__ bool better(float v, int i, float w, int j) { return (v > w) | ((v == w) & (i < j)); }

// Order-preserving map of a float (no NaN) onto unsigned integers, and back.
__device__ __forceinline__ uint32_t float_key(float v) {
    const uint32_t u = __float_as_uint(v);
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
__device__ __forceinline__ float key_float(uint32_t k) {
    return __uint_as_float((k & 0x80000000u) ? (k & 0x7fffffffu) : ~k);
}

__device__ __forceinline__ void fold_max_sum(float &m, float &s, const float2 &ms) {
    if (ms.x > m) {
        s = s * __expf(m - ms.x) + ms.y;   // exp(-inf) = 0 on the first tile
        m = ms.x;
    } else if (ms.x > -INFINITY) {
        s += ms.y * __expf(ms.x - m);
    }
}

// One partial list as it was written by the head GEMM, best first.
template <int kLen>
struct TileList {
    float2 ms;
    float v[kLen];
    int i[kLen];
};

template <int kLen>
__device__ __forceinline__ void load_list(TileList<kLen> &l, const MergeArgs &g, size_t tile, bool valid) {
    l.ms = make_float2(-INFINITY, 0.0f);
    if (valid) {
        l.ms = __ldcg((const float2 *)g.part_ms + tile);
        if constexpr (kLen == 2) {
            const float2 v = __ldcg((const float2 *)g.part_val + tile);
            const int2 i = __ldcg((const int2 *)g.part_idx + tile);
            l.v[0] = v.x; l.v[1] = v.y;
            l.i[0] = i.x; l.i[1] = i.y;
        } else if constexpr (kLen == 4) {
            const float4 v = __ldcg((const float4 *)g.part_val + tile);
            const int4 i = __ldcg((const int4 *)g.part_idx + tile);
            l.v[0] = v.x; l.v[1] = v.y; l.v[2] = v.z; l.v[3] = v.w;
            l.i[0] = i.x; l.i[1] = i.y; l.i[2] = i.z; l.i[3] = i.w;
        } else {
            const Float8 v = ldcg8(g.part_val + 8 * tile), i = ldcg8((const float *)g.part_idx + 8 * tile);
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                l.v[q] = v.v[q];
                l.i[q] = __float_as_int(i.v[q]);
            }
        }
    }
}

// What merge_select leaves in every warp of the group: lane j < rounds holds the j-th best entry of the row
// (-inf / 0x7fffffff when there are fewer), all lanes its log-sum-exp.
struct MergeOut {
    float val;
    int id;
    float lse;
};

// The `rounds` best entries (rounds <= kMaxRounds) of row r's partial lists and the row's log-sum-exp.  kLen: the lists' slots
// (list_slots).
// The step is a chain of latencies in a kernel that runs for a few microseconds, so it has one barrier and little
// code: thread t takes the lists t, t + kThreads, ... one at a time (they are sorted best first), and its warp extracts
// its own `rounds` best with warp-wide integer reductions (redux.sync: maximum of the value keys, then minimum token id
// among the lanes that hold it), carrying the winners of the lists so far as one more entry of lanes 0 .. rounds - 1.
// After the barrier every warp merges the warps' sorted results, one head per lane, in `rounds` more rounds, so that
// no second barrier is needed.  143 lists of a 16-row level: 5.2 us for the whole kernel with a running list of eight
// folded per thread and block-wide rounds (three times the code), 3.6 now; the last level with its prune 10.4 -> 7.1 (7B
// shape), 13.5 -> 9.3 (13B).
// `meanwhile` runs while the first lists are in flight.
struct Nothing {
    __device__ __forceinline__ void operator()() const {}
};
template <int kThreads, int kLen, typename Sync, typename Meanwhile = Nothing>
__device__ __forceinline__ MergeOut merge_select(const MergeArgs &g, int r, int tid, Scratch *sc, int rounds,
                                                 Meanwhile meanwhile = Meanwhile()) {
    constexpr int kWarps = kThreads / 32;
    static_assert(kWarps <= kMaxGroupWarps, "scratch arrays");
    const int lane = tid & 31, warp = tid >> 5;
    const int n_tiles = g.n_tiles, len = g.list_len > 0 ? g.list_len : g.topk;   // valid slots of every list
    const size_t first = (size_t)r * n_tiles;

    float cv = -INFINITY;   // the warp's winners so far: lane j the j-th
    int ci = 0x7fffffff;
    float m = -INFINITY, s = 0.0f;
    TileList<kLen> next;
    load_list(next, g, first + tid, tid < n_tiles);
    meanwhile();
    for (int t0 = warp * 32; t0 < n_tiles; t0 += kThreads) {   // (uniform over the warp)
        const TileList<kLen> cur = next;
        const bool valid = t0 + lane < n_tiles;
        load_list(next, g, first + t0 + kThreads + lane, t0 + kThreads + lane < n_tiles);
        fold_max_sum(m, s, cur.ms);
        float tv[kLen];
        int ti[kLen];
#pragma unroll
        for (int q = 0; q < kLen; ++q) {
            tv[q] = cur.v[q];
            ti[q] = cur.i[q];
        }
#pragma unroll
        for (int j = 0; j < kLen; ++j) {
            const bool none = (j >= len) | !valid;   // slots past the list's length hold nothing
            tv[j] = none ? -INFINITY : tv[j];
            ti[j] = none ? 0x7fffffff : ti[j];
        }
        float nv = -INFINITY;
        int ni = 0x7fffffff;
#pragma unroll 1
        for (int j = 0; j < rounds; ++j) {
            const bool carried = better(cv, ci, tv[0], ti[0]);
            const float hv = carried ? cv : tv[0];
            const int hi = carried ? ci : ti[0];
            const uint32_t key = float_key(hv);
            const uint32_t bk = __reduce_max_sync(0xffffffffu, key);
            const int bi = (int)__reduce_min_sync(0xffffffffu, key == bk ? (uint32_t)hi : 0xffffffffu);
            const bool mine = (key == bk) & (hi == bi);   // token ids are unique, so one lane owns a real entry
            const bool pop = mine & !carried;
            cv = mine & carried ? -INFINITY : cv;
            ci = mine & carried ? 0x7fffffff : ci;
#pragma unroll
            for (int q = 0; q < kLen - 1; ++q) {
                tv[q] = pop ? tv[q + 1] : tv[q];
                ti[q] = pop ? ti[q + 1] : ti[q];
            }
            tv[kLen - 1] = pop ? -INFINITY : tv[kLen - 1];
            ti[kLen - 1] = pop ? 0x7fffffff : ti[kLen - 1];
            nv = lane == j ? key_float(bk) : nv;
            ni = lane == j ? bi : ni;
        }
        cv = nv;
        ci = ni;
    }
    // the warp's (max, sum-exp)
    float wm = m;
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) wm = fmaxf(wm, __shfl_xor_sync(0xffffffffu, wm, off));
    float ws = (m > -INFINITY) ? s * __expf(m - wm) : 0.0f;
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) ws += __shfl_xor_sync(0xffffffffu, ws, off);
    MergeOut out;
    if constexpr (kWarps == 1) {   // nothing to merge (`sc` is not used)
        out.val = cv;
        out.id = ci;
        out.lse = wm + logf(ws);
        return out;
    }
    if (lane < rounds) {
        sc->cand_k[warp][lane] = float_key(cv);
        sc->cand_i[warp][lane] = ci;
    }
    if (lane == 0) {
        sc->red_m[warp] = wm;
        sc->red_s[warp] = ws;
    }
    Sync::sync();
    {
        const float pm = lane < kWarps ? sc->red_m[lane] : -INFINITY;
        const float ps = lane < kWarps ? sc->red_s[lane] : 0.0f;
        float bm = pm;
#pragma unroll
        for (int off = kMaxGroupWarps / 2; off > 0; off >>= 1) bm = fmaxf(bm, __shfl_xor_sync(0xffffffffu, bm, off));
        float bs = pm > -INFINITY ? ps * __expf(pm - bm) : 0.0f;
#pragma unroll
        for (int off = kMaxGroupWarps / 2; off > 0; off >>= 1) bs += __shfl_xor_sync(0xffffffffu, bs, off);
        out.lse = __shfl_sync(0xffffffffu, bm + logf(bs), 0);
    }
    out.val = -INFINITY;
    out.id = 0x7fffffff;
    const uint32_t none_key = float_key(-INFINITY);
    uint32_t hk = lane < kWarps ? sc->cand_k[lane][0] : none_key;
    uint32_t hi = lane < kWarps ? (uint32_t)sc->cand_i[lane][0] : 0x7fffffffu;
    int used = 0;
#pragma unroll 1
    for (int j = 0; j < rounds; ++j) {
        const uint32_t bk = __reduce_max_sync(0xffffffffu, hk);
        const uint32_t bi = __reduce_min_sync(0xffffffffu, hk == bk ? hi : 0xffffffffu);
        if (lane == j) {
            out.val = key_float(bk);
            out.id = (int)bi;
        }
        if (lane < kWarps && hk == bk && hi == bi) {
            ++used;
            hk = used < rounds ? sc->cand_k[lane][used] : none_key;
            hi = used < rounds ? (uint32_t)sc->cand_i[lane][used] : 0x7fffffffu;
        }
    }
    return out;
}

// The rows of the next level's embedding table that the children's gather is about to read, requested into L2 as soon
// as their tokens are known: the gather is the next kernel's first dependent load and goes to DRAM otherwise.
template <int kThreads>
__device__ __forceinline__ void prefetch_embeddings(const MergeArgs &g, const MergeOut &o, int tid) {
    if (g.next_emb == nullptr) return;
    for (int j = 0; j < g.topk; ++j) {
        const int t = __shfl_sync(0xffffffffu, o.id, j);
        if (t < 0 || t >= g.next_emb_rows) continue;
        const char *row = (const char *)g.next_emb + (size_t)t * g.next_emb_bytes;
        for (int i = tid * 128; i < g.next_emb_bytes; i += kThreads * 128)
            asm volatile("prefetch.global.L2 [%0];" ::"l"(row + i));
    }
}

// The row's top-k tokens and log-probabilities become its children.  `writer` = false: another CTA writes them.
template <int kThreads, int kLen, typename Sync, typename Meanwhile = Nothing>
__device__ __forceinline__ MergeOut merge_expand_row(const MergeArgs &g, int r, int tid, Scratch *sc, bool writer = true,
                                                     Meanwhile meanwhile = Meanwhile()) {
    const float base = (tid < g.topk && g.score_in && !g.lse_out) ? __ldcg(g.score_in + r) : 0.0f;   // in flight during the merge
    const MergeOut o = merge_select<kThreads, kLen, Sync>(g, r, tid, sc, g.topk, meanwhile);
    if (writer && tid < g.topk) {
        g.tok_out[(size_t)r * g.topk + tid] = o.id;
        g.score_out[(size_t)r * g.topk + tid] = g.lse_out ? o.val : base + (o.val - o.lse);
    }
    if (g.lse_out != nullptr && tid == 0) g.lse_out[r] = o.lse;
    prefetch_embeddings<kThreads>(g, o, tid);
    return o;
}

// The kBatch children of one parent row, all at once: gather + mix + LayerNorm + exact GELU (Sec. 3.1: siblings share the
// projected parent state and differ in the token embedding).
// Lane j of every warp holds child j's token (`tok`, as merge_select returns it), `first_child` is the row of child 0
// in the next level.  The projected parent state (sum of the split-K partials, added in
// ascending order) and the LayerNorm parameters are loaded once; the children's embedding rows
// are requested together and the two LayerNorm reductions are done for all of them with one barrier
// each (red_a / red_b: kThreads / 32 x kBatch floats each).  d <= 8 * kThreads * kIters, d % 8 == 0.
template <int kThreads, int kIters, int kBatch, typename Sync>
__device__ __forceinline__ void mix_children(const MixArgs &m, int parent, int first_child, int tok, float *red_a, float *red_b,
                                             int tid) {
    constexpr int kWarps = kThreads / 32;
    const int d = m.d, lane = tid & 31, warp = tid >> 5;
    float pv[kIters][8], gv[kIters][8], bv[kIters][8];
#pragma unroll
    for (int it = 0; it < kIters; ++it) {
        const int i = (it * kThreads + tid) * 8;
        const int ic = i < d ? i : 0;
#pragma unroll
        for (int j = 0; j < 8; ++j) pv[it][j] = 0.0f;
        if (i < d) {
            const float *p = m.P + (size_t)parent * d + i;
            for (int sp = 0; sp < m.p_splits; ++sp) {
                const Float8 x = ldcg8(p + sp * m.p_split_stride);
#pragma unroll
                for (int j = 0; j < 8; ++j) pv[it][j] += x.v[j];
            }
        }
        const float4 g0 = *(const float4 *)(m.gamma + ic), g1 = *(const float4 *)(m.gamma + ic + 4);
        const float4 b0 = *(const float4 *)(m.beta + ic), b1 = *(const float4 *)(m.beta + ic + 4);
        gv[it][0] = g0.x; gv[it][1] = g0.y; gv[it][2] = g0.z; gv[it][3] = g0.w;
        gv[it][4] = g1.x; gv[it][5] = g1.y; gv[it][6] = g1.z; gv[it][7] = g1.w;
        bv[it][0] = b0.x; bv[it][1] = b0.y; bv[it][2] = b0.z; bv[it][3] = b0.w;
        bv[it][4] = b1.x; bv[it][5] = b1.y; bv[it][6] = b1.z; bv[it][7] = b1.w;
    }
    float h[kBatch][kIters][8];
    float part[kBatch];
    uint4 ev[kBatch][kIters];
#pragma unroll
    for (int q = 0; q < kBatch; ++q) {
        const int t = __shfl_sync(0xffffffffu, tok, q);
        const bool tok_ok = t >= 0 && t < m.V;
        if (!tok_ok && tid == 0) report_error(m.err, SPEC_ERR_TOKEN_RANGE);
#pragma unroll
        for (int it = 0; it < kIters; ++it) {
            const int i = (it * kThreads + tid) * 8;
            ev[q][it] = make_uint4(0u, 0u, 0u, 0u);
            if (tok_ok && i < d) ev[q][it] = *(const uint4 *)(m.emb + (size_t)t * d + i);
        }
    }
#pragma unroll
    for (int q = 0; q < kBatch; ++q) {
        part[q] = 0.0f;
#pragma unroll
        for (int it = 0; it < kIters; ++it) {
            const int i = (it * kThreads + tid) * 8;
            const uint32_t ew[4] = {ev[q][it].x, ev[q][it].y, ev[q][it].z, ev[q][it].w};
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const float z = (j & 1) ? __uint_as_float(ew[j >> 1] & 0xffff0000u) : __uint_as_float(ew[j >> 1] << 16);
                h[q][it][j] = i < d ? mix_element(m, pv[it][j], z) : 0.0f;
                part[q] += h[q][it][j];
            }
        }
    }
    // batch-wide reductions: warp shuffles, one slot per (warp, child), then every thread adds the warps' slots
    float mean[kBatch], rstd[kBatch];
#pragma unroll
    for (int pass = 0; pass < 2; ++pass) {
        float *red = pass == 0 ? red_a : red_b;
#pragma unroll
        for (int q = 0; q < kBatch; ++q) {
            float v = part[q];
#pragma unroll
            for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
            if (lane == 0) red[warp * kBatch + q] = v;
        }
        Sync::sync();
#pragma unroll
        for (int q = 0; q < kBatch; ++q) {
            float t = 0.0f;
#pragma unroll
            for (int w = 0; w < kWarps; ++w) t += red[w * kBatch + q];
            if (pass == 0) {
                mean[q] = t / (float)d;
                part[q] = 0.0f;
#pragma unroll
                for (int it = 0; it < kIters; ++it) {
                    const int i = (it * kThreads + tid) * 8;
                    if (i < d) {
#pragma unroll
                        for (int j = 0; j < 8; ++j) {
                            const float c = h[q][it][j] - mean[q];
                            part[q] += c * c;
                        }
                    }
                }
            } else {
                rstd[q] = rsqrtf(t / (float)d + m.eps);
            }
        }
    }
#pragma unroll
    for (int q = 0; q < kBatch; ++q) {
        const size_t row = (size_t)first_child + q;
#pragma unroll
        for (int it = 0; it < kIters; ++it) {
            const int i = (it * kThreads + tid) * 8;
            uint32_t packed[4];
#pragma unroll
            for (int j = 0; j < 8; j += 4) {
                float4 y;
                y.x = (h[q][it][j] - mean[q]) * rstd[q] * gv[it][j] + bv[it][j];
                y.y = (h[q][it][j + 1] - mean[q]) * rstd[q] * gv[it][j + 1] + bv[it][j + 1];
                y.z = (h[q][it][j + 2] - mean[q]) * rstd[q] * gv[it][j + 2] + bv[it][j + 2];
                y.w = (h[q][it][j + 3] - mean[q]) * rstd[q] * gv[it][j + 3] + bv[it][j + 3];
                y = gelu_erf4(y);
                packed[j >> 1] = pack_bf16x2(y.x, y.y);
                packed[(j >> 1) + 1] = pack_bf16x2(y.z, y.w);
            }
            if (i < d) *(uint4 *)(m.S_out + row * d + i) = make_uint4(packed[0], packed[1], packed[2], packed[3]);
        }
    }
}

struct __align__(8) LeafKey {
    float score;
    int leaf;
};

__device__ __forceinline__ bool leaf_before(const LeafKey &a, const LeafKey &b) {
    return (a.score > b.score) | ((a.score == b.score) & (a.leaf < b.leaf));
}

// Writes candidate `rank` of sequence b: its score and the tokens on the path from the root to `leaf`.
__device__ __forceinline__ void emit_candidate(const PruneArgs &pa, int L, int K, int32_t *cand_tok, float *cand_logp,
                                               int b, int rank, float score, int leaf) {
    cand_logp[(size_t)b * K + rank] = score;
    int idx = leaf;            // index among this sequence's nodes of level n
    int per_seq = L;           // nodes of this sequence at level l + 1
    for (int l = pa.n - 1; l >= 0; --l) {
        cand_tok[((size_t)b * K + rank) * pa.n + l] = __ldcg(pa.tok[l] + (size_t)b * per_seq + idx);
        idx /= pa.topk[l];
        per_seq /= pa.topk[l];
    }
}

// Tokens on the path from the root to `leaf` of sequence b, requested together (their addresses depend on the
// leaf index only, not on one another).
__device__ __forceinline__ void load_path(const PruneArgs &pa, int L, int b, int leaf, int32_t (&path)[SPEC_MAX_HEADS]) {
    int idx = leaf, per_seq = L;
#pragma unroll
    for (int l = SPEC_MAX_HEADS - 1; l >= 0; --l) {
        if (l < pa.n) {
            path[l] = __ldcg(pa.tok[l] + (size_t)b * per_seq + idx);
            idx /= pa.topk[l];
            per_seq /= pa.topk[l];
        }
    }
}

// Leaves of one sequence as integers: the order-preserving image of the score above 4095 - leaf, so that the greater key
// is the better leaf and no two are equal.  (+ 0.0f: -0 and +0 are equal.)
static_assert(SPEC_MAX_LEAVES <= 4096, "twelve bits for the leaf");
__device__ __forceinline__ uint64_t leaf_key(float score, int leaf) {
    return ((uint64_t)float_key(score + 0.0f) << 12) | (uint32_t)(4095 - leaf);
}

// The K best (K <= kSelectMax) of the L keys in shared memory, to `sel` in any order: a radix selection from the top, eight
// bits a pass, until the keys of the bin that holds the K-th are wanted all or none.  `hist`: 256 words, `state`: 4 words.
constexpr int kSelectMax = 256;
constexpr int kSelectWords = 256 + 4 + 2 * kSelectMax;   // 32-bit words behind the keys: histogram, state, selection
template <int kThreads, typename Sync>
__device__ __forceinline__ void select_leaves(const uint64_t *keys, int L, int K, uint32_t *hist, uint32_t *state,
                                              uint64_t *sel, int tid) {
    const int lane = tid & 31, warp = tid >> 5;
    uint64_t prefix = 0;   // the keys still in question are those whose bits from `top` on equal it
    int top = 44, need = K;
    while (true) {
        const int shift = top > 8 ? top - 8 : 0;
        for (int i = tid; i < 256; i += kThreads) hist[i] = 0;
        if (tid == 0) state[3] = 0;
        Sync::sync();
        for (int i0 = warp * 32; i0 < L; i0 += kThreads) {   // (uniform over the warp)
            const uint64_t k = i0 + lane < L ? keys[i0 + lane] : 0;
            const bool in = i0 + lane < L && (k >> top) == prefix;
            // scores crowd in few bins: one addition per bin and warp
            const uint32_t bin = in ? (uint32_t)(k >> shift) & ((1u << (top - shift)) - 1u) : 256u;
            const uint32_t peers = __match_any_sync(0xffffffffu, bin);
            if (in && lane == __ffs(peers) - 1) atomicAdd(hist + bin, __popc(peers));
        }
        Sync::sync();
        if (warp == 0) {   // lane l: bins 255 - 8 l downwards
            uint32_t c[8], sum = 0;
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                c[q] = hist[255 - 8 * lane - q];
                sum += c[q];
            }
            uint32_t upto = sum;
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
                const uint32_t o = __shfl_up_sync(0xffffffffu, upto, off);
                if (lane >= off) upto += o;
            }
            uint32_t above = upto - sum;
            if (above < (uint32_t)need && upto >= (uint32_t)need) {
#pragma unroll
                for (int q = 0; q < 8; ++q) {
                    if (above < (uint32_t)need && above + c[q] >= (uint32_t)need) {
                        state[0] = 255 - 8 * lane - q;
                        state[1] = need - above;
                        state[2] = c[q];
                    }
                    above += c[q];
                }
            }
        }
        Sync::sync();
        prefix = (prefix << (top - shift)) | state[0];
        top = shift;
        need = (int)state[1];
        if (need == (int)state[2] || top == 0) break;
    }
    const uint64_t least = prefix << top;
    for (int i = tid; i < L; i += kThreads)
        if (keys[i] >= least) sel[atomicAdd(state + 3, 1u)] = keys[i];
    Sync::sync();
}

// Sequence b: the K best leaves by (score desc, leaf index asc), traced back to the root.  `keys`:
// shared memory for Lpad entries, Lpad the power of two >= max(L, 2), and kSelectWords more when L > 256.  Up to 256 leaves
// every thread counts how many leaves precede its own (that is its rank; no barriers) and has requested the tokens of its
// own leaves' paths together with the scores, so a kept leaf is written out without another trip to memory.  Of longer lists
// the K best are selected first and then ranked among themselves (2016 rows, 1512 leaves, K = 3: the last kernel 63 us with a
// sort, 15.8 so); only when more than 256 are kept the whole list is sorted.
template <int kThreads, typename Sync>
__device__ __forceinline__ void prune_sequence(const float *leaf_score, const PruneArgs &pa, int L, int Lpad, int K,
                                               int32_t *cand_tok, float *cand_logp, int b, int tid, LeafKey *keys) {
    constexpr int kOwn = (256 + kThreads - 1) / kThreads;   // leaves per thread in the ranked form
    int32_t path[kOwn][SPEC_MAX_HEADS];
    if (L <= 256) {
#pragma unroll
        for (int q = 0; q < kOwn; ++q)
            if (tid + q * kThreads < L) load_path(pa, L, b, tid + q * kThreads, path[q]);
    }
    if (L > 256 && K <= kSelectMax) {
        uint64_t *k64 = (uint64_t *)keys;
        uint32_t *hist = (uint32_t *)(keys + Lpad), *state = hist + 256;
        uint64_t *sel = (uint64_t *)(state + 4);
        for (int i = tid; i < L; i += kThreads) k64[i] = leaf_key(__ldcg(leaf_score + (size_t)b * L + i), i);
        select_leaves<kThreads, Sync>(k64, L, K, hist, state, sel, tid);   // (begins with a barrier)
        for (int i = tid; i < K; i += kThreads) {
            const uint64_t mine = sel[i];
            const int leaf = 4095 - (int)(mine & 4095u);
            int32_t own[SPEC_MAX_HEADS];
            load_path(pa, L, b, leaf, own);
            int rank = 0;
            for (int j = 0; j < K; ++j) rank += sel[j] > mine ? 1 : 0;
            cand_logp[(size_t)b * K + rank] = __ldcg(leaf_score + (size_t)b * L + leaf);
#pragma unroll
            for (int l = 0; l < SPEC_MAX_HEADS; ++l)
                if (l < pa.n) cand_tok[((size_t)b * K + rank) * pa.n + l] = own[l];
        }
        return;
    }
    Sync::sync();   // a previous call may still be reading the keys
    for (int i = tid; i < Lpad; i += kThreads) {
        keys[i].score = (i < L) ? __ldcg(leaf_score + (size_t)b * L + i) : -INFINITY;
        keys[i].leaf = i < L ? i : 0x7fffffff;
    }
    Sync::sync();
    if (L <= 256) {
#pragma unroll
        for (int q = 0; q < kOwn; ++q) {
            const int i = tid + q * kThreads;
            if (i >= L) continue;
            const LeafKey mine = keys[i];
            int rank = 0;
            for (int j = 0; j < L; ++j) rank += leaf_before(keys[j], mine) ? 1 : 0;
            if (rank < K) {
                cand_logp[(size_t)b * K + rank] = mine.score;
#pragma unroll
                for (int l = 0; l < SPEC_MAX_HEADS; ++l)
                    if (l < pa.n) cand_tok[((size_t)b * K + rank) * pa.n + l] = path[q][l];
            }
        }
        return;
    }
    for (int size = 2; size <= Lpad; size <<= 1) {
        for (int stride = size >> 1; stride > 0; stride >>= 1) {
            for (int i = tid; i < Lpad / 2; i += kThreads) {
                const int lo = 2 * i - (i & (stride - 1));
                const int hi = lo + stride;
                const bool ascending_block = ((lo & size) == 0);   // "ascending" = best first
                const LeafKey x = keys[lo], y = keys[hi];
                const bool swap = ascending_block ? leaf_before(y, x) : leaf_before(x, y);
                if (swap) {
                    keys[lo] = y;
                    keys[hi] = x;
                }
            }
            Sync::sync();
        }
    }
    for (int k = tid; k < K; k += kThreads)
        emit_candidate(pa, L, K, cand_tok, cand_logp, b, k, keys[k].score, keys[k].leaf);
}

// Shared memory of prune_sequence.
inline size_t prune_smem_bytes(int L, int Lpad) {
    return sizeof(LeafKey) * (size_t)Lpad + (L > 256 ? sizeof(uint32_t) * kSelectWords : 0);
}

// Prune folded into the kernel that writes the last level.  Every row's CTA makes its children visible
// (fence), then counts itself in for its sequence; the CTA that brings the count to rows_per_seq sees all
// of the sequence's leaves and prunes it.  No CTA ever waits for another.  `flag`: one shared int.
template <int kThreads, typename Sync>
__device__ __forceinline__ void prune_if_last(const MergeArgs &g, int r, int tid, LeafKey *keys, int *flag) {
    if (g.seq_done == nullptr) return;
    const int b = r / g.rows_per_seq;
    if (g.rows_per_seq > 1) {   // (a sequence of one row is complete with this CTA's own children)
        __threadfence();        // this CTA's children before its count
        Sync::sync();
        if (tid == 0) *flag = (atomicAdd(g.seq_done + b, 1) == g.rows_per_seq - 1) ? 1 : 0;
        Sync::sync();
        if (*flag == 0) return;
        __threadfence();        // the other CTAs' children after the last count
    } else {
        Sync::sync();
    }
    prune_sequence<kThreads, Sync>(g.score_out, g.prune, g.L, g.Lpad, g.K, g.cand_tok, g.cand_logp, b, tid, keys);
}

}  // namespace rows
}  // namespace spec
