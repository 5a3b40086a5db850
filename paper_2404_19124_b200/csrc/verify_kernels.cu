// Greedy multi-candidate verification (Sec. 1, Sec. 3.1, Sec. 5 of arXiv 2404.19124):
// a bandwidth-bound streaming arg-max over every row of the base model's logits followed by
// the longest-matching-prefix / best-candidate reduction.
//
// Everywhere the tensor is one run of 16-byte vectors, whatever the row length and the alignment of its base: positions
// are elements counted from the 16-byte boundary at or below the base, a row is a partial vector (read element by
// element), a run of whole vectors, and another partial vector.  A lane keeps eight 128-bit streaming loads in flight.  For
// bf16 the running maximum is taken on packed pairs (max.bf16x2) and the element index is only resolved when a vector
// beats the lane's current best, so the common case costs about one ALU operation per element.
//
// Three forms (one_kernel_form and pool_form choose):
//   verify_seq_kernel    one CTA per sequence does the whole job: its warps take equal contiguous ranges of the sequence's
//                        vectors, fold them into a (value, index) key per row in shared memory, and the CTA accepts.
//   verify_pool_kernel + verify_accept_kernel    long rows: two ranges of vectors per SM, each shared out among the warps of a CTA
//   verify_stream_kernel + verify_accept_kernel    all vectors cut into equal contiguous ranges, one per warp, a single
//                        wave over the whole GPU; a row that lies in one range is finished there, of the others every
//                        piece leaves a (value, index) partial; one CTA per sequence folds those and accepts.
#include <float.h>

#include <mutex>

#include "spec_common.cuh"

namespace spec {

namespace {

constexpr int kArgmaxThreads = 256;
constexpr int kWarpsPerBlock = kArgmaxThreads / 32;
constexpr int kIdxNone = 0x7fffffff;
constexpr int kSeqThreads = 1024;
constexpr int kSeqMaxRows = 4000;   // 47 KB of keys and table

__device__ __forceinline__ uint32_t max_bf16x2(uint32_t a, uint32_t b) {
    uint32_t d;
    asm("max.bf16x2 %0, %1, %2;" : "=r"(d) : "r"(a), "r"(b));   // a NaN operand is dropped
    return d;
}

__device__ __forceinline__ uint4 ld_stream(const uint4 *p) {
    uint4 v;
    asm volatile("ld.global.nc.L1::no_allocate.v4.u32 {%0,%1,%2,%3}, [%4];"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
                 : "l"(p));
    return v;
}

// best/idx: the lane's running (maximum, first index).  `base` is the index of element 0 of v.
__device__ __forceinline__ void consume_bf16(const uint4 &v, int base, float &best, int &idx) {
    uint32_t m2 = max_bf16x2(max_bf16x2(v.x, v.y), max_bf16x2(v.z, v.w));
    float mx = fmaxf(__uint_as_float(m2 << 16), __uint_as_float(m2 & 0xffff0000u));
    if (mx > best) {   // rare after the first few vectors
        best = mx;
        const uint32_t w[4] = {v.x, v.y, v.z, v.w};
        int pos = 7;
#pragma unroll
        for (int i = 3; i >= 0; --i) {
            if (__uint_as_float(w[i] & 0xffff0000u) == mx) pos = 2 * i + 1;
            if (__uint_as_float(w[i] << 16) == mx) pos = 2 * i;
        }
        idx = base + pos;
    }
}

__device__ __forceinline__ void consume_f32(const uint4 &v, int base, float &best, int &idx) {
    const float f[4] = {__uint_as_float(v.x), __uint_as_float(v.y), __uint_as_float(v.z), __uint_as_float(v.w)};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        if (f[i] > best) {
            best = f[i];
            idx = base + i;
        }
    }
}

// (value desc, index asc) combine across the warp.
__device__ __forceinline__ void warp_argmax(float &best, int &idx) {
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        float ob = __shfl_xor_sync(0xffffffffu, best, off);
        int oi = __shfl_xor_sync(0xffffffffu, idx, off);
        const bool take = (ob > best) | ((ob == best) & (oi < idx));
        best = take ? ob : best;
        idx = take ? oi : idx;
    }
}

constexpr int kStreamUnroll = 8;

// Elements per vector and its logarithm.
template <bool kBf16>
struct Elem {
    static constexpr int kEpv = kBf16 ? 8 : 4, kShift = kBf16 ? 3 : 2;
    static __device__ __forceinline__ float load(const char *base, long long i) {
        return kBf16 ? bf16_bits_to_float(((const uint16_t *)base)[i]) : ((const float *)base)[i];
    }
};

// The n vectors at `src`, the first of which is element col0 of its row, read by `kGroup` threads of which this is number t.
template <bool kBf16, int kGroup>
__device__ __forceinline__ void scan_vectors(const uint4 *src, int n, int col0, int t, float &best, int &idx) {
    for (int i = t; i < n; i += kGroup * kStreamUnroll) {
        uint4 v[kStreamUnroll];
#pragma unroll
        for (int u = 0; u < kStreamUnroll; ++u)
            if (i + kGroup * u < n) v[u] = ld_stream(src + i + kGroup * u);
#pragma unroll
        for (int u = 0; u < kStreamUnroll; ++u) {
            if (i + kGroup * u < n) {
                const int col = col0 + (i + kGroup * u) * Elem<kBf16>::kEpv;
                if (kBf16) consume_bf16(v[u], col, best, idx);
                else consume_f32(v[u], col, best, idx);
            }
        }
    }
}

// The part of a row (elements [rs, re) of the run of vectors at `base`) that lies in vectors [a, e), read by `kGroup`
// threads of which this is number `t`: the thread's maximum and its first index within the row.
template <bool kBf16, int kGroup>
__device__ __forceinline__ void scan_row(const char *base, long long rs, long long re, long long a, long long e, int t,
                                         float &best, int &idx) {
    using E = Elem<kBf16>;
    const long long hv = rs >> E::kShift, body0 = (rs + E::kEpv - 1) >> E::kShift, body1 = re >> E::kShift;
    if (body0 != hv && hv >= a && hv < e) {   // the row starts inside a vector
        const long long i = rs + t, end = min(re, body0 << E::kShift);
        const float x = i < end ? E::load(base, i) : -INFINITY;
        if (x > best) {
            best = x;
            idx = t;
        }
    }
    const long long p = max(body0, a), q = min(body1, e);
    if (q > p) {
        scan_vectors<kBf16, kGroup>((const uint4 *)base + p, (int)(q - p), (int)((p << E::kShift) - rs), t, best, idx);
    }
    if (body1 >= body0 && body1 >= a && body1 < e && (re & (E::kEpv - 1)) != 0) {   // ... and ends inside another
        const long long i = (body1 << E::kShift) + t;
        const float x = i < re ? E::load(base, i) : -INFINITY;
        if (x > best) {
            best = x;
            idx = (int)(i - rs);
        }
    }
}

// (value, first index) as one integer whose maximum is the arg-max: the order-preserving image of the value above the
// complement of the index.  0 stands for "nothing above -inf".  (+ 0.0f: -0 and +0 are equal.)
__device__ __forceinline__ uint32_t value_key(float v) {
    const uint32_t u = __float_as_uint(v + 0.0f);
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
__device__ __forceinline__ unsigned long long argmax_key(float v, int idx) {
    return idx == kIdxNone ? 0ull : ((unsigned long long)value_key(v) << 32) | (uint32_t)~idx;
}
// The index that a key stands for (0 where a row has no value above -inf), and the key as a partial.
__device__ __forceinline__ int key_index(unsigned long long k) { return k == 0ull ? 0 : (int)~(uint32_t)k; }
__device__ __forceinline__ float2 key_partial(unsigned long long k) {
    const uint32_t hi = (uint32_t)(k >> 32);
    return k == 0ull ? make_float2(-INFINITY, __int_as_float(kIdxNone))
                     : make_float2(__uint_as_float((hi & 0x80000000u) ? (hi & 0x7fffffffu) : ~hi), __int_as_float(key_index(k)));
}

// Places of the partials.  A border between two warps is crossed by one row at most, so the pieces behind a border are
// numbered by their warp; a row's first piece goes to a place of its row or of its warp behind those, whichever are fewer.
__host__ __device__ __forceinline__ long long first_piece(long long warps, int rows, int row, long long w) {
    return warps + (rows < warps ? row : w);
}

// vec_per_warp vectors per warp, `warps` of them at most; row r is elements [skew + r * V, + V).
template <bool kBf16>
__global__ void __launch_bounds__(kArgmaxThreads, 4)
verify_stream_kernel(const char *__restrict__ base, int skew, int rows, int V, long long total_vec, int vec_per_warp,
                     int warps, int32_t *g_out, float2 *part) {
    griddep_launch();
    griddep_wait();
    using E = Elem<kBf16>;
    const int lane = threadIdx.x & 31;
    const long long w = (long long)blockIdx.x * kWarpsPerBlock + (threadIdx.x >> 5);
    const long long beg = w * vec_per_warp, end = min(total_vec, beg + vec_per_warp);
    if (beg >= end) return;
    const long long first = (beg << E::kShift) - skew;
    for (int row = first > 0 ? (int)(first / V) : 0; row < rows; ++row) {
        const long long rs = skew + (long long)row * V;
        if ((rs >> E::kShift) >= end) break;
        float best = -INFINITY;
        int idx = kIdxNone;
        scan_row<kBf16, 32>(base, rs, rs + V, beg, end, lane, best, idx);
        warp_argmax(best, idx);
        if (lane == 0) {
            const bool begins = (rs >> E::kShift) >= beg, ends = ((rs + V - 1) >> E::kShift) < end;   // in this range
            if (begins && ends) g_out[row] = idx == kIdxNone ? 0 : idx;   // (nothing above -inf, all NaN: 0)
            else part[begins ? first_piece(warps, rows, row, w) : w] = make_float2(best, __int_as_float(idx));
        }
    }
}

// Long rows: two CTAs per SM take one range of vectors each, and a CTA's warps take blocks of its range as they get to them.  Bound
// by DRAM.  Of the four CTAs that an SM holds in the form above one is served last, trip after trip (its first loads return after
// 10 us, the others' after 3), so that in the end it runs on alone; here its warps take fewer blocks instead.  The keys of the
// rows that a range touches gather in shared memory, so that few pieces are left to the accept kernel, and most trips end with
// one comparison against their row's key.  14 warps of 64 registers: one CTA fits beside a CTA of the head GEMM, as a CTA of the
// form above does, so that a draft on another stream and a verification do not shut each other out (one CTA of 28 warps an SM:
// the two together at the 7B shape 135.0 us a pair -> 137.0, so 135.1; at batch 4 with fp32 logits the verification 47 -> 64, so
// 46), and two leave the accept kernel's CTAs their place: they are there when the last block is read.
constexpr int kPoolThreads = 448, kPoolPerSm = 2, kPoolMaxRows = 128;

template <bool kBf16>
__global__ void __maxnreg__(64)
verify_pool_kernel(const char *__restrict__ base, int skew, int rows, int V, long long total_vec, int vec_per_cta, int block,
                   int ctas, int32_t *g_out, float2 *part) {
    __shared__ unsigned long long keys[kPoolMaxRows];
    __shared__ int taken;
    using E = Elem<kBf16>;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const long long beg = (long long)blockIdx.x * vec_per_cta, end = min(total_vec, beg + vec_per_cta);
    const long long first = (beg << E::kShift) - skew;
    const int row0 = first > 0 ? (int)(first / V) : 0, n = (int)(end - beg);
    const int into = (int)(first - (long long)row0 * V);   // the range begins this many elements into row0 (-skew: before it)
    griddep_launch();
    for (int i = threadIdx.x; i < kPoolMaxRows; i += kPoolThreads) keys[i] = 0ull;
    if (threadIdx.x == 0) taken = kPoolThreads / 32 * block;
    __syncthreads();
    griddep_wait();
    // the whole vectors of every row (positions below are relative to the range)
    for (int a = warp * block; a < n;) {
        int next = 0;
        if (lane == 0) next = atomicAdd(&taken, block);
        const int e = min(a + block, n), at = into + (a << E::kShift);
        int r = at > 0 ? (int)((uint32_t)at / (uint32_t)V) : 0;
        for (int re = (r + 1) * V - into;; ++r, re += V) {   // re: where the row ends, in elements from the range's start
            const int rs = re - V;
            const int p = max(a, (rs + E::kEpv - 1) >> E::kShift), q = min(e, re >> E::kShift);
            for (int i = p; i < q; i += 32 * kStreamUnroll) {
                const uint4 *src = (const uint4 *)base + beg;
                uint4 v[kStreamUnroll];
#pragma unroll
                for (int u = 0; u < kStreamUnroll; ++u) v[u] = ld_stream(src + min(i + 32 * u + lane, q - 1));
                // What the row has already, as one lane sees it: other warps raise the key meanwhile, and whether the warp goes on
                // to the next reduction must be one decision.  (An old value costs an update, the maximum is taken there.)
                uint32_t seen = 0u;
                if (lane == 0) seen = (uint32_t)(*(volatile unsigned long long *)&keys[r] >> 32);
                seen = __shfl_sync(0xffffffffu, seen, 0);
                float mx;
                if (kBf16) {
                    uint32_t m[kStreamUnroll];
#pragma unroll
                    for (int u = 0; u < kStreamUnroll; ++u) m[u] = max_bf16x2(max_bf16x2(v[u].x, v[u].y), max_bf16x2(v[u].z, v[u].w));
#pragma unroll
                    for (int h = kStreamUnroll / 2; h > 0; h >>= 1)
#pragma unroll
                        for (int u = 0; u < h; ++u) m[u] = max_bf16x2(m[u], m[u + h]);
                    mx = fmaxf(__uint_as_float(m[0] << 16), __uint_as_float(m[0] & 0xffff0000u));
                } else {
                    float m[kStreamUnroll];
#pragma unroll
                    for (int u = 0; u < kStreamUnroll; ++u)
                        m[u] = fmaxf(fmaxf(__uint_as_float(v[u].x), __uint_as_float(v[u].y)), fmaxf(__uint_as_float(v[u].z), __uint_as_float(v[u].w)));
#pragma unroll
                    for (int h = kStreamUnroll / 2; h > 0; h >>= 1)
#pragma unroll
                        for (int u = 0; u < h; ++u) m[u] = fmaxf(m[u], m[u + h]);
                    mx = m[0];
                }
                const uint32_t key = mx > -INFINITY ? value_key(mx) : 0u;   // (NaN: nothing)
                const uint32_t top = __reduce_max_sync(0xffffffffu, key);
                if (top == 0u || top < seen) continue;   // most trips find nothing that reaches what their row has already
                int pos = kIdxNone;
                if (key == top) {
#pragma unroll
                    for (int u = kStreamUnroll - 1; u >= 0; --u) {
                        const uint32_t w[4] = {v[u].x, v[u].y, v[u].z, v[u].w};
                        const int at_u = min(i + 32 * u + lane, q - 1) << E::kShift;
#pragma unroll
                        for (int h = 3; h >= 0; --h) {
                            if (kBf16) {
                                if (__uint_as_float(w[h] & 0xffff0000u) == mx) pos = at_u + 2 * h + 1;
                                if (__uint_as_float(w[h] << 16) == mx) pos = at_u + 2 * h;
                            } else if (__uint_as_float(w[h]) == mx) {
                                pos = at_u + h;
                            }
                        }
                    }
                }
                pos = __reduce_min_sync(0xffffffffu, pos);
                if (lane == 0) atomicMax(&keys[r], ((unsigned long long)top << 32) | (uint32_t)~(pos - rs));
            }
            if ((re >> E::kShift) >= e || row0 + r + 1 >= rows) break;
        }
        a = __shfl_sync(0xffffffffu, next, 0);
    }
    // the vectors that rows share: lanes 0 to kEpv - 1 take the row's first elements, the next ones its last
    for (int r = warp; row0 + r < rows && (r * V - into) >> E::kShift < n; r += kPoolThreads / 32) {
        const int rs = r * V - into, re = rs + V;
        const int head = min((rs + E::kEpv - 1) >> E::kShift << E::kShift, re), tail = max(re >> E::kShift << E::kShift, head);
        const int i = lane < E::kEpv ? rs + lane : tail + lane - E::kEpv;
        const bool mine = lane < E::kEpv ? i < head : lane < 2 * E::kEpv && i < re;
        const int vec = i >> E::kShift;
        const float x = mine && vec >= 0 && vec < n ? E::load(base + (beg << 4), i) : -INFINITY;
        const uint32_t key = x > -INFINITY ? value_key(x) : 0u;
        const uint32_t top = __reduce_max_sync(0xffffffffu, key);
        const int pos = __reduce_min_sync(0xffffffffu, key == top ? i - rs : kIdxNone);
        if (lane == 0 && top != 0u) atomicMax(&keys[r], ((unsigned long long)top << 32) | (uint32_t)~pos);
    }
    __syncthreads();
    for (int i = threadIdx.x;; i += kPoolThreads) {
        const int row = row0 + i;
        const long long rs = skew + (long long)row * V;
        if (row >= rows || (rs >> E::kShift) >= end) break;
        const bool begins = (rs >> E::kShift) >= beg, ends = ((rs + V - 1) >> E::kShift) < end;   // in this range
        if (begins && ends) g_out[row] = key_index(keys[i]);
        else part[begins ? first_piece(ctas, rows, row, blockIdx.x) : (long long)blockIdx.x] = key_partial(keys[i]);
    }
}

// (Everything an earlier kernel of the stream wrote - the partials, the candidates, the match lengths and the
// indices spec_next_ctx consumes - is read with ld.global.cg, never through the non-coherent path: these
// kernels start early under programmatic dependent launch and the same addresses are rewritten call after call.
// base_logits itself is streamed with ld.global.nc: it must be complete before the call is enqueued behind
// its producer on the stream, which stream order guarantees.)
// Tokens of one candidate, at most SPEC_MAX_HEADS of them, requested together.
__device__ __forceinline__ void load_candidate(const int32_t *cand_tok, size_t c, int n, bool valid,
                                               int32_t (&tok)[SPEC_MAX_HEADS]) {
#pragma unroll
    for (int j = 0; j < SPEC_MAX_HEADS; ++j) tok[j] = valid && j < n ? __ldcg(cand_tok + c * n + j) : -1;
}

// Sequence b's acceptance from its arg-max table (K * (n + 1) entries, visible to the whole CTA), by a CTA whose threads
// hold the tokens of their first candidate in `ctok`.  `key_s`: shared, zero.
__device__ __forceinline__ void accept_sequence(const int32_t *cand_tok, const int32_t *gtab, int b, int K, int n,
                                                int32_t (&ctok)[SPEC_MAX_HEADS], unsigned int *key_s,
                                                int32_t *accept_len, int32_t *best_cand, int32_t *next_tok) {
    for (int k = threadIdx.x; k < K; k += blockDim.x) {
        const int32_t *gk = gtab + k * (n + 1);
        if (k != (int)threadIdx.x) load_candidate(cand_tok, (size_t)b * K + k, n, true, ctok);   // more candidates than threads
        int m = 0;
        bool open = true;
#pragma unroll
        for (int j = 0; j < SPEC_MAX_HEADS; ++j) {
            open = open && j < n && ctok[j] == gk[j];
            m += open ? 1 : 0;
        }
        if (open && n > SPEC_MAX_HEADS) {   // longer candidates than the registers hold: one token at a time
            const int32_t *c = cand_tok + ((size_t)b * K + k) * n;
            while (m < n && __ldcg(c + m) == gk[m]) ++m;
        }
        // longest prefix first, then the lowest candidate index
        atomicMax(key_s, ((unsigned)m << 16) | (unsigned)(0xffff - k));
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        const int m = (int)(*key_s >> 16), k = 0xffff - (int)(*key_s & 0xffffu);
        accept_len[b] = m;
        best_cand[b] = k;
        next_tok[b] = gtab[k * (n + 1) + m];
    }
}

__global__ void __launch_bounds__(128)
verify_accept_kernel(const int32_t *cand_tok, const float2 *part, int K, int n, int V, int skew, int shift, int rows, int warps,
                     int vec_per_warp, int32_t *g_out, int g_in_smem, int32_t *accept_len, int32_t *best_cand,
                     int32_t *next_tok, int32_t *err) {
    // The sequence's arg-max table is re-read by other threads for the prefix match: from shared memory
    // when it fits the default 48 KB, otherwise from the copy in g_out this CTA has just written (global
    // writes of a CTA are visible to its own threads after the barrier).
    extern __shared__ int32_t g_s[];   // [K * (n + 1)] if g_in_smem
    __shared__ unsigned int key_s;
    const int b = blockIdx.x, rows_b = K * (n + 1);
    griddep_launch();
    if (threadIdx.x == 0) key_s = 0u;
    griddep_wait();
    if (threadIdx.x == 0 && b == 0 && err != nullptr) *err = 0;
    // The step is a handful of dependent round trips to L2, so every load that does not depend on another is
    // requested before the first one is used: the tokens of this thread's first candidate now, a row's partials
    // eight slots at a time.
    constexpr int kBatch = 8;
    int32_t ctok[SPEC_MAX_HEADS];
    load_candidate(cand_tok, (size_t)b * K + threadIdx.x, n, (int)threadIdx.x < K, ctok);
    for (int r = threadIdx.x; r < rows_b; r += blockDim.x) {
        const size_t gr = (size_t)b * rows_b + r;
        // the row's pieces are the warps whose ranges its vectors touch
        const long long rs = skew + (long long)gr * V, v0 = rs >> shift, v1 = (rs + V - 1) >> shift;
        const bool narrow = (v1 >> 32) == 0;
        const long long w0 = narrow ? (uint32_t)v0 / (uint32_t)vec_per_warp : v0 / vec_per_warp;
        const int chunks = (int)((narrow ? (uint32_t)v1 / (uint32_t)vec_per_warp : v1 / vec_per_warp) - w0) + 1;
        const float2 *first = part + first_piece(warps, rows, (int)gr, w0), *rest = part + w0;
        const int whole = __ldcg(g_out + gr);   // (what it says only if the row was finished where it was read)
        float best = -INFINITY;
        int arg = 0;   // a row without any value above -inf (all NaN) yields 0
        for (int c0 = 0; c0 < chunks; c0 += kBatch) {
            float2 v[kBatch];
#pragma unroll
            for (int j = 0; j < kBatch; ++j) v[j] = c0 + j < chunks && chunks > 1 ? __ldcg(c0 + j == 0 ? first : rest + c0 + j) : make_float2(-INFINITY, 0.0f);
#pragma unroll
            for (int j = 0; j < kBatch; ++j) {
                const bool take = v[j].x > best;   // chunks ascend, so the first maximum wins
                best = take ? v[j].x : best;
                arg = take ? __float_as_int(v[j].y) : arg;
            }
        }
        if (chunks == 1) arg = whole;
        else g_out[gr] = arg;
        if (g_in_smem) g_s[r] = arg;
    }
    __syncthreads();
    accept_sequence(cand_tok, g_in_smem ? g_s : g_out + (size_t)b * rows_b, b, K, n, ctok, &key_s, accept_len, best_cand,
                    next_tok);
}

// ---- one CTA per sequence ---------------------------------------------------------------------------

template <bool kBf16>
__global__ void __launch_bounds__(kSeqThreads, 1)
verify_seq_kernel(const char *__restrict__ base, int skew, const int32_t *cand_tok, int K, int n, int V,
                  int32_t *g_out, int32_t *accept_len, int32_t *best_cand, int32_t *next_tok, int32_t *err) {
    extern __shared__ unsigned long long keys[];   // [K * (n + 1)], then the arg-max table, int32 [K * (n + 1)]
    __shared__ unsigned int key_s;
    using E = Elem<kBf16>;
    const int rows_b = K * (n + 1), lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int b = blockIdx.x;
    int32_t *g_s = (int32_t *)(keys + rows_b);
    griddep_launch();
    for (int r = threadIdx.x; r < rows_b; r += kSeqThreads) keys[r] = 0ull;
    if (threadIdx.x == 0) key_s = 0u;
    __syncthreads();
    griddep_wait();
    if (threadIdx.x == 0 && blockIdx.x == 0 && err != nullptr) *err = 0;
    int32_t ctok[SPEC_MAX_HEADS];
    load_candidate(cand_tok, (size_t)b * K + threadIdx.x, n, (int)threadIdx.x < K, ctok);
    // the sequence as a run of vectors of its own
    const long long s0 = skew + (long long)b * rows_b * V;
    const char *seq = base + ((s0 >> E::kShift) << 4);
    const int rel = (int)(s0 & (E::kEpv - 1));
    const long long total = (rel + (long long)rows_b * V + E::kEpv - 1) >> E::kShift;
    constexpr int kWarps = kSeqThreads / 32;
    const long long per = (total + kWarps - 1) / kWarps;
    const long long beg = (long long)warp * per, end = min(total, beg + per);
    if (beg < end) {
        const long long first = (beg << E::kShift) - rel;
        for (int row = first > 0 ? (int)(first / V) : 0; row < rows_b; ++row) {
            const long long rs = rel + (long long)row * V;
            if ((rs >> E::kShift) >= end) break;
            float best = -INFINITY;
            int idx = kIdxNone;
            scan_row<kBf16, 32>(seq, rs, rs + V, beg, end, lane, best, idx);
            warp_argmax(best, idx);
            if (lane == 0) atomicMax(&keys[row], argmax_key(best, idx));
        }
    }
    __syncthreads();
    for (int r = threadIdx.x; r < rows_b; r += kSeqThreads) {
        const int arg = key_index(keys[r]);
        g_s[r] = arg;
        g_out[(size_t)b * rows_b + r] = arg;
    }
    __syncthreads();
    accept_sequence(cand_tok, g_s, b, K, n, ctok, &key_s, accept_len, best_cand, next_tok);
}

// ---- early-exit form ------------------------------------------------------------------------------
// The rows of a candidate matter only up to its first mismatch (Sec. 1: the tokens after a rejected
// one are discarded), so reading them is optional work: one CTA or a cluster of them per candidate walks its rows in order,
// takes the arg-max of a row together (a contiguous part each, eight 128-bit loads in flight per thread) and stops
// after the first row whose arg-max differs from the speculated token.  Bytes read fall from
// B K (n+1) V to sum over candidates of (m + 1) V elements; rows that were not read get g = -1.
__device__ __forceinline__ uint32_t cluster_rank() {
    uint32_t r;
    asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ void cluster_barrier() {
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
constexpr int kMaxEarlyCtas = 8;

template <bool kBf16>
__global__ void __launch_bounds__(kArgmaxThreads)
verify_early_kernel(const char *__restrict__ base, const int32_t *cand_tok, int n, int V, int ctas, int32_t *g,
                    int32_t *match_len, int32_t *best_cand, int32_t *next_tok, int32_t *err) {
    // One barrier per row: every warp hands its key to every CTA of the cluster, in one of two sets of slots by turns (a set
    // is written again only after the next row's barrier, when all its readers have arrived).
    __shared__ unsigned long long keys[2][kMaxEarlyCtas * kWarpsPerBlock];
    using E = Elem<kBf16>;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int rank = ctas > 1 ? (int)cluster_rank() : 0, c = blockIdx.x / ctas, slots = ctas * kWarpsPerBlock;
    griddep_launch();
    if (ctas > 1) cluster_barrier();   // the other CTAs' shared memory is there
    griddep_wait();
    const int row_vec = V >> E::kShift, per = (row_vec + ctas - 1) / ctas;   // a row is a run of whole vectors
    const int first = rank * per, count = min(row_vec - first, per);
    int m = n, j = 0, last = 0;
    for (; j <= n; ++j) {
        const long long row = (long long)c * (n + 1) + j;
        const int tok = j < n ? __ldcg(cand_tok + (size_t)c * n + j) : -1;
        float best = -INFINITY;
        int idx = kIdxNone;
        scan_vectors<kBf16, kArgmaxThreads>((const uint4 *)base + row * row_vec + first, count, first * E::kEpv, tid, best, idx);
        warp_argmax(best, idx);
        unsigned long long *set = keys[j & 1];
        if (lane < ctas) {
            const unsigned long long key = argmax_key(best, idx);
            if (ctas > 1) {
                uint32_t there;
                asm volatile("mapa.shared::cluster.u32 %0, %1, %2;"
                             : "=r"(there)
                             : "r"((uint32_t)__cvta_generic_to_shared(set + rank * kWarpsPerBlock + warp)), "r"(lane));
                asm volatile("st.shared::cluster.u64 [%0], %1;" ::"r"(there), "l"(key) : "memory");
            } else {
                set[warp] = key;
            }
        }
        if (ctas > 1) cluster_barrier();
        else __syncthreads();
        unsigned long long k = lane < slots ? set[lane] : 0ull;
        if (slots > 32) k = max(k, set[lane + 32 < slots ? lane + 32 : lane]);
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) k = max(k, __shfl_xor_sync(0xffffffffu, k, off));
        const int arg = key_index(k);   // a row without any value above -inf (all NaN) yields 0
        last = arg;
        if (rank == 0 && tid == 0) g[row] = arg;
        if (j < n && tok != arg) {   // uniform over the cluster
            m = j;
            break;
        }
    }
    if (rank == 0) {
        for (int jj = j + 1 + tid; jj <= n; jj += kArgmaxThreads) g[(size_t)c * (n + 1) + jj] = -1;
        if (tid == 0) match_len[c] = m;
        if (best_cand != nullptr && tid == 0) {   // one candidate per sequence: it is the best, m its accepted length
            best_cand[c] = 0;
            next_tok[c] = last;
            if (c == 0 && err != nullptr) *err = 0;
        }
    }
}

// One CTA per sequence: the candidate with the longest match (lowest index among equals) and its bonus token.
__global__ void __launch_bounds__(128)
verify_accept_early_kernel(const int32_t *g, const int32_t *match_len, int K, int n, int32_t *accept_len,
                           int32_t *best_cand, int32_t *next_tok, int32_t *err) {
    __shared__ unsigned int key_s;
    griddep_launch();
    griddep_wait();
    const int b = blockIdx.x;
    if (threadIdx.x == 0) {
        key_s = 0u;
        if (b == 0 && err != nullptr) *err = 0;
    }
    __syncthreads();
    for (int k = threadIdx.x; k < K; k += blockDim.x)
        atomicMax(&key_s, ((unsigned)__ldcg(match_len + (size_t)b * K + k) << 16) | (unsigned)(0xffff - k));
    __syncthreads();
    if (threadIdx.x == 0) {
        const int m = (int)(key_s >> 16), k = 0xffff - (int)(key_s & 0xffffu);
        accept_len[b] = m;
        best_cand[b] = k;
        next_tok[b] = __ldcg(g + ((size_t)b * K + k) * (n + 1) + m);
    }
}

size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

}  // namespace

// One kernel when a sequence is little enough for one CTA to read in less time than a second kernel costs.  One CTA reads
// about 65 GB/s: 64 KB 4.9 us per call against 6.8 us in two kernels (both bound by the host), 256 KB 7.6 against 9.5 alone
// but 65.0 against 63.6 us inside a decoding step, 512 KB 11.6 against 9.7, 1 MB 15.3 against 9.5.
// Its CTA has an SM to itself, so that more sequences than SMs take turns of about 3.3 us, while the two-kernel form reads them all
// in one wave; that one walks the rows of a warp's range one by one, about 0.8 us each (256 vectors hold 8 * 256 / V rows of bf16),
// and is the slower the shorter the rows.  us per call, one kernel / two, four candidates of four rows: V 64, 444 sequences
// 10.6 / 39.7, 1000 23.9 / 41.9, 3000 69 / 44; V 256, 256 7.2 / 13.1, 444 10.6 / 11.2, 1000 24 / 16; V 1024, 148 4.6 / 6.5,
// 149 7.3 / 6.4, 1000 25.8 / 13.9; V 4096, 148 5.8 / 8.5, 149 10.1 / 8.4, 1000 40.6 / 24.8.
constexpr long long kSeqMaxBytes = 128 << 10;
bool one_kernel_form(int B, int rows_b, int V, int dtype) {
    const long long turns = ((long long)B + num_sms() - 1) / num_sms();
    return rows_b <= kSeqMaxRows && (long long)rows_b * V * (dtype == SPEC_BF16 ? 2 : 4) <= kSeqMaxBytes &&
           (turns - 1) * V <= 64 * (dtype == SPEC_BF16 ? Elem<true>::kEpv : Elem<false>::kEpv);
}

// Where verify_pool_kernel takes over from verify_stream_kernel: up to 1 GB in all; from 25 MB where rows have 48 KB or more, from
// 4.8 MB for rows of 60 KB, from 1.9 MB for rows of 188 KB, of which the other form leaves dozens of pieces to the accept kernel.
// Measured behind matrix products that fill the GPU to its power limit, as a base model's last layer does (a call with its
// launches), and in a loop of calls; pool / stream:
//   rows, bf16   5 MB   8 MB   16 MB   33 MB   65 MB   131 MB   262 MB   400 MB   800 MB   1.5 GB   3 GB
//   47-48 KB     1.16   1.02   0.97    0.92    0.92    0.97     0.97     0.97     0.95     1.00     1.00
//   62 KB        1.02   0.98   0.93    0.92    0.93    0.97     0.97     0.97     0.94     1.00     1.00
//   98 KB        0.99   0.90   0.87    0.87    0.93    0.96     0.96     0.97     0.89     0.91     1.01
//   250 KB       0.87   0.81   0.76    0.83    0.90    0.96     0.95     0.93     0.94     0.98     0.99
// (A loop of calls gains about the same, down to the 8 MB where the host's 7.3 us for two launches are what it takes.)  fp32: 48 KB
// 1.15 at 8 MB, 1.03 at 16, 0.99 at 33; 125 KB 0.94 to 1.00 up to 16 MB, 0.93 at 33.  Shorter rows, bf16: 31 KB 0.99 at 16 MB,
// 0.94 at 33 and 65, 1.00 to 1.02 at 131 and 200; 16 KB no better at most sizes (a trip ends at a row's end).
constexpr long long kPoolMinRowVec = 3072, kPoolMaxRowVec = 1 << 24, kPoolMaxVec = 64 << 20;
long long pool_min_vec(long long row_vec) { return row_vec >= 12000 ? 120000 : row_vec >= 3840 ? 300000 : 1536 << 10; }
bool pool_form(long long total_vec, long long row_vec) {
    return row_vec >= kPoolMinRowVec && row_vec <= kPoolMaxRowVec && total_vec >= pool_min_vec(row_vec) && total_vec <= kPoolMaxVec &&
           (total_vec / (kPoolPerSm * num_sms()) + 1) / row_vec + 3 <= kPoolMaxRows;
}

// Resident CTAs per SM of the streaming kernel (launch bound above) times the SM count gives the
// number of warps of one full wave; every warp gets an equal range of at least one unrolled trip.
VerifyPlan make_verify_plan(int B, int K, int n, int V, int dtype) {
    VerifyPlan p{};
    p.rows = B * K * (n + 1);
    const int epv = dtype == SPEC_BF16 ? 8 : 4;
    const long long total = ((long long)p.rows * V + 2 * epv - 2) / epv;   // vectors, the base at its least aligned
    const long long wave_warps = (long long)num_sms() * 4 * kWarpsPerBlock;
    long long c = (total + wave_warps - 1) / wave_warps;
    if (c < 32 * kStreamUnroll) c = 32 * kStreamUnroll;
    if (c > (1ll << 30)) c = 1ll << 30;
    p.vec_per_warp = (int)c;
    p.warps = (int)((total + c - 1) / c);
    p.off_g = kWsAlign;   // (the scratch is sized for the form that leaves most pieces)
    p.off_part = align_up(p.off_g + sizeof(int32_t) * (size_t)p.rows, kWsAlign);
    // at most a partial behind every border and a first piece for every row that crosses one.  Never less than 4 bytes per
    // candidate, the early-exit form's match lengths.
    const size_t partials = sizeof(float2) * ((size_t)p.warps + (p.rows < p.warps ? p.rows : p.warps));
    const size_t lengths = sizeof(int32_t) * (size_t)B * K;
    p.total = align_up(p.off_part + (partials > lengths ? partials : lengths), kWsAlign);
    if (pool_form(total, V / epv)) {
        const long long ctas = (long long)kPoolPerSm * num_sms(), range = (total + ctas - 1) / ctas;
        p.pool = true;
        p.vec_per_warp = (int)range;
        p.warps = (int)((total + range - 1) / range);
    }
    return p;
}

int launch_verify(const int32_t *cand_tok, const void *base_logits, int dtype, int B, int K, int n, int V,
                  int32_t *accept_len, int32_t *best_cand, int32_t *next_tok, void *ws, const VerifyPlan &plan,
                  cudaStream_t st) {
    char *w = (char *)ws;
    int32_t *err = (int32_t *)w;
    int32_t *g = (int32_t *)(w + plan.off_g);
    const bool bf16 = dtype == SPEC_BF16;
    const int shift = bf16 ? 3 : 2, esz = bf16 ? 2 : 4;
    const char *base = (const char *)((uintptr_t)base_logits & ~(uintptr_t)15);
    const int skew = (int)(((uintptr_t)base_logits & 15) / esz), rows_b = K * (n + 1);
    if (one_kernel_form(B, rows_b, V, dtype)) {
        const size_t smem = (sizeof(unsigned long long) + sizeof(int32_t)) * (size_t)rows_b;
        SPEC_CUDA_TRY(launch_pdl(bf16 ? verify_seq_kernel<true> : verify_seq_kernel<false>, dim3((unsigned)B), dim3(kSeqThreads),
                                 smem, st, base, skew, cand_tok, K, n, V, g, accept_len, best_cand, next_tok, err));
        return SPEC_OK;
    }
    float2 *part = (float2 *)(w + plan.off_part);
    const long long total = (skew + (long long)plan.rows * V + (1 << shift) - 1) >> shift;
    const long long warps = (total + plan.vec_per_warp - 1) / plan.vec_per_warp;
    if (plan.pool) {
        // Blocks of up to five trips, of which a warp gets a whole number, so that the warps end together; short ones where there
        // are many of them.  us a call in blocks of one / two / four trips and so, V 32000 in bf16 behind a matrix product: 25 MB
        // (1.5 trips a warp) 19.1 / 17.6 / 19.4, 17.6; 47 MB 23.0 / 22.1 / 21.6, 21.6; 65 MB 26.8 / 24.6 / 23.6, 23.6; 76 MB
        // 29.8 / 27.6 / 28.6, 25.7; 131 MB 38.4 / 34.0 / 33.8, 33.8; 400 MB 84.1 / 73.7 / 74.7, 73.7.
        const int trips = (plan.vec_per_warp / (kPoolThreads / 32) + 32 * kStreamUnroll - 1) / (32 * kStreamUnroll);
        const int turns = (trips + 4) / 5, block = 32 * kStreamUnroll * (trips > 20 ? 2 : (trips + turns - 1) / turns);
        SPEC_CUDA_TRY(launch_pdl(bf16 ? verify_pool_kernel<true> : verify_pool_kernel<false>, dim3((unsigned)warps),
                                 dim3(kPoolThreads), 0, st, base, skew, plan.rows, V, total, plan.vec_per_warp, block, plan.warps, g,
                                 part));
    } else {
        const unsigned grid = (unsigned)((warps + kWarpsPerBlock - 1) / kWarpsPerBlock);
        SPEC_CUDA_TRY(launch_pdl(bf16 ? verify_stream_kernel<true> : verify_stream_kernel<false>, dim3(grid), dim3(kArgmaxThreads),
                                 0, st, base, skew, plan.rows, V, total, plan.vec_per_warp, plan.warps, g, part));
    }
    size_t smem = sizeof(int32_t) * (size_t)rows_b;
    const int g_in_smem = smem <= 40 * 1024;
    if (!g_in_smem) smem = 0;
    SPEC_CUDA_TRY(launch_pdl(verify_accept_kernel, dim3(B), dim3(128), smem, st, cand_tok, (const float2 *)part, K, n, V, skew,
                             shift, plan.rows, plan.warps, plan.vec_per_warp, g, g_in_smem, accept_len, best_cand, next_tok, err));
    return SPEC_OK;
}

// CTAs per candidate of the early-exit form: as many as the GPU holds at once (four per SM), up to eight, and no more than
// leave each of them three 16-byte vectors per thread of a row.  One CTA reads a row at 30 GB/s, whatever else the GPU does.
// us per call for 1 / 2 / 4 / 8 CTAs, bf16, match lengths uniform: V 128256, 8 candidates 43.2 / 27.8 / 18.9 / 14.0,
// 128 candidates 57.2 / 43.2 / 32.8 / 36.4, 256 candidates 56.4 / 42.1 / 44.1 / 51.5, 512 candidates 66.4 / 68.4 / 71.3 / 90.7
// (50 for the bytes; 69.2 with two barriers per row), 2048 candidates of two rows 120.0 / 127.0 / 153.5 / 215.7 (118.6 with
// two barriers); V 32000, 32 candidates 18.6 / 15.3 / 14.0 / 13.8; V 8000, 128 candidates 9.6 / 11.7 / 12.5 / 19.3.
int early_ctas(int candidates, int row_vec) {
    int ctas = 1;
    while (2 * ctas <= kMaxEarlyCtas && (long long)candidates * 2 * ctas <= 4ll * num_sms() &&
           row_vec >= 3 * kArgmaxThreads * 2 * ctas)
        ctas *= 2;
    return ctas;
}

// Early-exit form; returns SPEC_ERR_SHAPE when the rows are not whole 16-byte vectors (the caller then
// uses the streaming form).
int launch_verify_early(const int32_t *cand_tok, const void *base_logits, int dtype, int B, int K, int n, int V,
                        int32_t *accept_len, int32_t *best_cand, int32_t *next_tok, void *ws, const VerifyPlan &plan,
                        cudaStream_t st) {
    const bool bf16 = dtype == SPEC_BF16;
    if (V % (bf16 ? 8 : 4) != 0 || ((uintptr_t)base_logits % 16) != 0) return SPEC_ERR_SHAPE;
    char *w = (char *)ws;
    int32_t *err = (int32_t *)w;
    int32_t *g = (int32_t *)(w + plan.off_g);
    int32_t *match_len = (int32_t *)(w + plan.off_part);   // B * K words; the partial maxima's area is not used here
    // One candidate per sequence: nothing to choose, so no second kernel.  Four rows each, bf16, us per call: 2 sequences, V 8000
    // 7.7 -> 6.1; 32 sequences, V 32000 11.6 -> 9.4.
    const bool single = K == 1;
    const int ctas = early_ctas(B * K, V / (bf16 ? 8 : 4));
    SPEC_CUDA_TRY(launch_pdl_cluster(bf16 ? verify_early_kernel<true> : verify_early_kernel<false>, dim3(B * K * ctas),
                                     dim3(kArgmaxThreads), 0, ctas, st, (const char *)base_logits, cand_tok, n, V, ctas, g,
                                     single ? accept_len : match_len, single ? best_cand : nullptr, next_tok, err));
    if (single) return SPEC_OK;
    SPEC_CUDA_TRY(launch_pdl(verify_accept_early_kernel, dim3(B), dim3(128), 0, st, (const int32_t *)g,
                             (const int32_t *)match_len, K, n, accept_len, best_cand, next_tok, err));
    return SPEC_OK;
}

}  // namespace spec

// ---- spec_next_ctx: the state vector the next draft starts from (Sec. 3.1) ----------------------
namespace spec {
namespace {

// One CTA per sequence copies base_state[b, best_cand[b], accept_len[b], :] to ctx_state[b, :].  The two
// indices come from the verify kernels earlier in the stream, hence the dependency wait before they are read.
__global__ void __launch_bounds__(128)
next_ctx_kernel(const uint16_t *__restrict__ base_state, const int32_t *best_cand, const int32_t *accept_len, int K,
                int n, int d, int vec_ok, uint16_t *__restrict__ ctx_state, int32_t *err) {
    griddep_launch();
    griddep_wait();
    const int b = blockIdx.x;
    const int k = __ldcg(best_cand + b), m = __ldcg(accept_len + b);
    uint16_t *dst = ctx_state + (size_t)b * d;
    if (k < 0 || k >= K || m < 0 || m > n) {   // never read outside the tensor: the row becomes zero
        if (threadIdx.x == 0) report_error(err, SPEC_ERR_INDEX_RANGE);
        for (int i = threadIdx.x; i < d; i += blockDim.x) dst[i] = 0;
        return;
    }
    const uint16_t *src = base_state + (((size_t)b * K + k) * (n + 1) + m) * d;
    if (vec_ok) {
        const uint4 *s4 = reinterpret_cast<const uint4 *>(src);
        uint4 *d4 = reinterpret_cast<uint4 *>(dst);
        for (int i = threadIdx.x; i < d / 8; i += blockDim.x) d4[i] = s4[i];
    } else {
        for (int i = threadIdx.x; i < d; i += blockDim.x) dst[i] = src[i];
    }
}

}  // namespace
}  // namespace spec

extern "C" int spec_next_ctx(const void *base_state, const int32_t *best_cand, const int32_t *accept_len, int B, int K,
                             int n, int d_base, void *ctx_state, int32_t *err_word, void *cuda_stream) {
    using namespace spec;
    if (!base_state || !best_cand || !accept_len || !ctx_state) return SPEC_ERR_INVALID_ARG;
    if (B <= 0 || K <= 0 || n <= 0 || d_base <= 0) return SPEC_ERR_INVALID_ARG;
    if (((uintptr_t)base_state % 2) != 0 || ((uintptr_t)ctx_state % 2) != 0) return SPEC_ERR_INVALID_ARG;
    if (err_word && ((uintptr_t)err_word % 4) != 0) return SPEC_ERR_INVALID_ARG;
    const int vec_ok = (d_base % 8 == 0) && ((uintptr_t)base_state % 16) == 0 && ((uintptr_t)ctx_state % 16) == 0;
    SPEC_CUDA_TRY(launch_pdl(next_ctx_kernel, dim3((unsigned)B), dim3(128), 0, (cudaStream_t)cuda_stream,
                             (const uint16_t *)base_state, best_cand, accept_len, K, n, d_base, vec_ok,
                             (uint16_t *)ctx_state, err_word));
    return SPEC_OK;
}

// ---- spec_verify_static: the verify scratch lives in the library's own device image ------------
// For hosts that cannot give the library a workspace (all device memory already committed to their
// own pools, or no allocation allowed where this runs).  Inside host code the array's name is only a
// handle for the runtime, not a device address: the address each device mapped it to is asked for
// once per device with cudaGetSymbolAddress and that pointer is what the kernels receive.
static __device__ __align__(256) unsigned char g_verify_static_scratch[SPEC_VERIFY_STATIC_SCRATCH_BYTES];

namespace {
constexpr int kMaxDevices = 64;
std::mutex g_static_mutex;
void *g_static_ptr[kMaxDevices] = {};
}  // namespace

extern "C" int spec_verify_static(const int32_t *cand_tok, const void *base_logits, int logits_dtype, int B, int K,
                                  int n, int V, int32_t *accept_len, int32_t *best_cand, int32_t *next_tok,
                                  void *cuda_stream) {
    using namespace spec;
    if (!cand_tok || !base_logits || !accept_len || !best_cand || !next_tok) return SPEC_ERR_INVALID_ARG;
    if (B <= 0 || K <= 0 || n <= 0 || V <= 0) return SPEC_ERR_INVALID_ARG;
    if (logits_dtype != SPEC_BF16 && logits_dtype != SPEC_F32) return SPEC_ERR_INVALID_ARG;
    if (K > 65535 || (long long)K * (n + 1) > 12288 || n > 32767) return SPEC_ERR_SHAPE;
    if ((long long)B * K * (n + 1) > (1ll << 30)) return SPEC_ERR_SHAPE;
    if (((uintptr_t)base_logits % (logits_dtype == SPEC_BF16 ? 2 : 4)) != 0) return SPEC_ERR_INVALID_ARG;
    const VerifyPlan plan = make_verify_plan(B, K, n, V, logits_dtype);
    if (plan.total > (size_t)SPEC_VERIFY_STATIC_SCRATCH_BYTES) return SPEC_ERR_STATIC_SCRATCH;

    int dev = -1;
    SPEC_CUDA_TRY(cudaGetDevice(&dev));
    if (dev < 0 || dev >= kMaxDevices) return SPEC_ERR_NO_DEVICE;
    void *scratch = nullptr;
    {
        std::lock_guard<std::mutex> lock(g_static_mutex);
        if (g_static_ptr[dev] == nullptr) {
            // first call on this device (which is current): where did this device map the array?
            void *ptr = nullptr;
            SPEC_CUDA_TRY(cudaGetSymbolAddress(&ptr, g_verify_static_scratch));
            if (ptr == nullptr || ((uintptr_t)ptr % kWsAlign) != 0) return SPEC_ERR_WORKSPACE;
            g_static_ptr[dev] = ptr;
        }
        scratch = g_static_ptr[dev];
    }
    return launch_verify(cand_tok, base_logits, logits_dtype, B, K, n, V, accept_len, best_cand, next_tok, scratch, plan,
                         (cudaStream_t)cuda_stream);
}

