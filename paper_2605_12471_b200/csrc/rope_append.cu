// Fused RoPE(q), RoPE(k) + append(k, v) for one chunk.
//
// Section 2 of the paper: the new tokens' position identifiers continue from the chunk's
// absolute start, so the rotations line up with the original sequence; Figure "KV-Fold": the
// chunk's K/V are appended to the cache and earlier rows are left as they are.
//
// Numerics (the cache bits are a contract): theta = pos * inv_freq[j] in fp64, cos/sin in fp64,
// each rounded once to fp32; then per output two fp32 operations,
//     lo' = fma(x_lo, c, -(x_hi * s))      hi' = fma(x_hi, c, x_lo * s)
// with the cross product rounded first, and one round-to-nearest-even to the cache dtype.
// Values are copied verbatim.  All global accesses are 16-byte vectors.
#include "kvfold_internal.h"

namespace kvf {
namespace {

constexpr int kThreads = 512;  // every thread has one 16-byte item of a bf16 Llama-shaped token (320 rotated segments + 128 value segments)

template <typename T> struct Vec16;
template <> struct Vec16<float> {
    static constexpr int N = 4;
    static __device__ __forceinline__ void unpack(const uint4 &v, float (&x)[4]) {
        x[0] = __uint_as_float(v.x); x[1] = __uint_as_float(v.y); x[2] = __uint_as_float(v.z); x[3] = __uint_as_float(v.w);
    }
    static __device__ __forceinline__ void store(float *p, const float (&x)[4]) {
        *reinterpret_cast<float4 *>(p) = make_float4(x[0], x[1], x[2], x[3]);
    }
};
template <> struct Vec16<__nv_bfloat16> {
    static constexpr int N = 8;
    static __device__ __forceinline__ void unpack(const uint4 &v, float (&x)[8]) {
        const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            x[2 * i] = __uint_as_float(w[i] << 16);
            x[2 * i + 1] = __uint_as_float(w[i] & 0xFFFF0000u);
        }
    }
    static __device__ __forceinline__ void store(__nv_bfloat16 *p, const float (&x)[8]) {
        uint32_t w[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            uint32_t lo = __bfloat16_as_ushort(__float2bfloat16_rn(x[2 * i]));
            uint32_t hi = __bfloat16_as_ushort(__float2bfloat16_rn(x[2 * i + 1]));
            w[i] = lo | (hi << 16);
        }
        *reinterpret_cast<uint4 *>(p) = make_uint4(w[0], w[1], w[2], w[3]);
    }
};

__device__ __forceinline__ void rotate(float a, float b, float c, float s, float &ra, float &rb) {
    float cross_a = __fmul_rn(b, s);
    float cross_b = __fmul_rn(a, s);
    ra = __fmaf_rn(a, c, -cross_a);
    rb = __fmaf_rn(b, c, cross_b);
}

// kTok = tokens per CTA, kResident = CTAs of an SM (see launch_type).
template <typename T, bool INTERLEAVED, int kTok, int kResident>
__global__ void __launch_bounds__(kThreads, kResident) rope_append_kernel(const RopeAppendArgs a) {
    constexpr int VEC = Vec16<T>::N;
    __shared__ float2 cs[kTok][kMaxHalfDim];   // (cos, sin) per (token, pair)

    const int d = a.d, half = d / 2;
    const int n_tok_blocks = (a.n + kTok - 1) / kTok;      // (a.n: the longest chunk of the launch)
    const int b = blockIdx.y;      // cache of a batch (0 when there is one cache)
    const RowMap rows{a.page_tables ? a.page_tables[b] : a.page_table, a.capacity, a.page_elems, a.d};
    // (the per-cache arrays of a ragged batch were written by an earlier kernel of the stream: under
    // a dependent launch they are visible only after the wait)
    if (a.prefixes || a.pos0s) pdl_wait();
    const int64_t prefix = a.prefixes ? a.prefixes[b] : a.prefix;
    const int64_t pos0 = a.pos0s ? a.pos0s[b] : a.pos0;
    const int n = a.ns ? (int)a.ns[b] : a.n;               // tokens this cache folds

    pdl_launch_dependents();
    if ((int)blockIdx.x >= n_tok_blocks) {
        pdl_wait();   // the attention of the step before may still be reading these rows' tile
        // Clear value rows between the new end of the cache and the next key-tile boundary,
        // so that a zero probability never multiplies stale non-finite bits.
        const int vec_per_row = d / VEC;
        const int zero_rows = n == 0 ? 0 : a.prefixes ? (int)((kKvTile - (prefix + n) % kKvTile) % kKvTile) : a.zero_rows;
        const int64_t total = (int64_t)zero_rows * a.Hkv * vec_per_row;
        const int64_t start = ((int64_t)blockIdx.x - n_tok_blocks) * kThreads + threadIdx.x;
        const int64_t stride = (int64_t)(gridDim.x - n_tok_blocks) * kThreads;
        T *vp = reinterpret_cast<T *>(a.v_plane);
        for (int64_t i = start; i < total; i += stride) {
            int c = (int)(i % vec_per_row);
            int64_t t = i / vec_per_row;
            int g = (int)(t % a.Hkv);
            int64_t row = prefix + n + t / a.Hkv;
            *reinterpret_cast<uint4 *>(vp + rows.offset(g, row) + c * VEC) =
                make_uint4(0, 0, 0, 0);
        }
        return;
    }

    const int tok0 = blockIdx.x * kTok;
    const int ntok = min(kTok, n - tok0);
    if (ntok <= 0) return;                                  // a shorter member of a batch

    for (int idx = threadIdx.x; idx < ntok * half; idx += kThreads) {
        int t = idx / half, j = idx % half;
        double theta = (double)(pos0 + tok0 + t) * a.table.inv_freq[j];
        double sn, cn;
        sincos(theta, &sn, &cn);
        cs[t][j] = make_float2((float)cn, (float)sn);
    }
    const int64_t qoff = (int64_t)b * a.n * a.H * d, koff = (int64_t)b * a.n * a.Hkv * d;
    const T *q = reinterpret_cast<const T *>(a.q) + qoff;
    const T *k = reinterpret_cast<const T *>(a.k_new) + koff;
    const T *v = reinterpret_cast<const T *>(a.v_new) + koff;
    T *qr = reinterpret_cast<T *>(a.q_rot) + qoff;
    T *kp = reinterpret_cast<T *>(a.k_plane);
    T *vp = reinterpret_cast<T *>(a.v_plane);
    const int heads = a.H + (a.k_new ? a.Hkv : 0);     // (queries only when no keys are given: kvf_attend)

    // A thread takes the same 16-byte item of every token of the CTA (rotated segments of q and k, behind them the
    // value segments, verbatim copies): where it lies is worked out once, and the tokens' loads go out back to back.
    const int rot_chunks = INTERLEAVED ? d / VEC : half / VEC;       // vectors per row (interleaved) or per half row
    const int rot_items = heads * rot_chunks;
    const int v_chunks = d / VEC;
    const int items = rot_items + (a.v_new ? a.Hkv * v_chunks : 0);
    struct Item {
        bool value, query;
        int c, g, row_heads;                                   // vector in the row, query head or KV head, heads of a token
        const T *src;                                          // the first token's
    };
    auto item = [&](int idx) {
        Item m;
        m.value = idx >= rot_items;
        const int it = m.value ? idx - rot_items : idx, chunks = m.value ? v_chunks : rot_chunks;
        m.c = it % chunks;
        const int hh = it / chunks;
        m.query = !m.value && hh < a.H;
        m.g = m.value || m.query ? hh : hh - a.H;
        m.row_heads = m.query ? a.H : a.Hkv;
        m.src = (m.query ? q : m.value ? v : k) + ((int64_t)tok0 * m.row_heads + m.g) * d + m.c * VEC;
        return m;
    };
    // The inputs' lines are called into L2 while the kernel before still finishes; they are read, as everything else, behind the wait.
    // Cold inputs, us: 128 steps of 256 tokens under a window 2547 -> 2508, 15 077 tokens of 28 / 4 heads in chunks of 256 2613 -> 2568;
    // eight steps of 2048 tokens the same.
    if ((int)threadIdx.x < items) {
        const Item m = item(threadIdx.x);
#pragma unroll
        for (int t = 0; t < kTok; ++t)
            if (t < ntok) {
                const T *line = m.src + (int64_t)t * m.row_heads * d;
                asm volatile("prefetch.global.L2 [%0];" ::"l"(line));
                if (!INTERLEAVED && !m.value) asm volatile("prefetch.global.L2 [%0];" ::"l"(line + half));
            }
    }
    __syncthreads();
    pdl_wait();   // the table above needs nothing from earlier kernels; the writes below do

    float amax = 0.f;               // largest magnitude written (tracked only under a range limit, fp32 caches)
    const bool ranged = sizeof(T) == 4 && a.range_limit > 0.f;
    for (int idx = threadIdx.x; idx < items; idx += kThreads) {
        const Item m = item(idx);
        const bool value = m.value, query = m.query;
        const int c = m.c, g = m.g;
        const T *src = m.src;
        const int64_t src_step = (int64_t)m.row_heads * d;
        T *plane = value ? vp : kp;
        auto dst = [&](int t) { return (query ? qr + ((int64_t)(tok0 + t) * a.H + g) * d : plane + rows.offset(g, prefix + tok0 + t)) + c * VEC; };
        uint4 lo[kTok], hi[kTok];
#pragma unroll
        for (int t = 0; t < kTok; ++t)
            if (t < ntok) {
                lo[t] = *reinterpret_cast<const uint4 *>(src + t * src_step);
                if (!INTERLEAVED && !value) hi[t] = *reinterpret_cast<const uint4 *>(src + t * src_step + half);
            }
#pragma unroll
        for (int t = 0; t < kTok; ++t) {
            if (t >= ntok) break;
            T *to = dst(t);
            if (value) {
                *reinterpret_cast<uint4 *>(to) = lo[t];
                if (ranged)
                    amax = fmaxf(fmaxf(amax, fmaxf(fabsf(__uint_as_float(lo[t].x)), fabsf(__uint_as_float(lo[t].y)))),
                                 fmaxf(fabsf(__uint_as_float(lo[t].z)), fabsf(__uint_as_float(lo[t].w))));
                continue;
            }
            float x[VEC], r[VEC];
            Vec16<T>::unpack(lo[t], x);
            if (!INTERLEAVED) {
                float y[VEC], ry[VEC];
                Vec16<T>::unpack(hi[t], y);
#pragma unroll
                for (int e = 0; e < VEC; ++e) {
                    const float2 w = cs[t][c * VEC + e];
                    rotate(x[e], y[e], w.x, w.y, r[e], ry[e]);
                }
                Vec16<T>::store(to, r);
                Vec16<T>::store(to + half, ry);
                if (ranged) {
#pragma unroll
                    for (int e = 0; e < VEC; ++e) amax = fmaxf(amax, fabsf(ry[e]));
                }
            } else {
#pragma unroll
                for (int e = 0; e < VEC; e += 2) {
                    const float2 w = cs[t][(c * VEC + e) / 2];
                    rotate(x[e], x[e + 1], w.x, w.y, r[e], r[e + 1]);
                }
                Vec16<T>::store(to, r);
            }
            if (ranged) {
#pragma unroll
                for (int e = 0; e < VEC; ++e) amax = fmaxf(amax, fabsf(r[e]));
            }
        }
    }
    if (ranged && amax > a.range_limit) atomicCAS(a.status, 0, 7);
}

}  // namespace

template <typename T, int TOK, int RESIDENT>
static cudaError_t launch_tok(const RopeAppendArgs &a, bool interleaved, int batch, cudaStream_t s) {
    int blocks = (a.n + TOK - 1) / TOK;
    if (a.zero_rows > 0) {
        int64_t vecs = (int64_t)a.zero_rows * a.Hkv * (a.d / Vec16<T>::N);
        blocks += (int)((vecs + kThreads - 1) / kThreads);
    }
    auto kernel = interleaved ? rope_append_kernel<T, true, TOK, RESIDENT> : rope_append_kernel<T, false, TOK, RESIDENT>;
    return launch_pdl(kernel, dim3(blocks, batch), dim3(kThreads), 0, s, a);
}

// One token per CTA while two CTAs on an SM hold the launch: a step waits for a token's chain (sines, loads, stores), and as a
// dependent launch no more than two to an SM are better than the four that 32 registers allow - they start while SMs are still taken
// and would crowd on the others (128 steps of 256 tokens under a window: 2994 us with two, 3077 with four).  More tokens: bf16
// four CTAs of one token on an SM, from seven tokens an SM on four tokens per CTA, which pay for the chain once; fp32
// two.  Members of a batch with fewer tokens than that keep one per CTA.  us per launch, cold inputs, plain launches back to
// back: bf16, 32 / 8 heads, one token with two / four CTAs on an SM, two, four tokens: 256 tokens 4.0 / 3.9 / 4.2 / 5.3; 360: 6.2 / 4.4 /
// 5.2 / 5.6; 512: 6.7 / 5.0 / 5.3 / 5.9; 640: 8.0 / 6.0 / 7.4 / 8.2; 1024: 10.9 / 8.0 / 9.1 / 8.3; 2048: 18.9 / 13.3 / 15.5 / 14.3; 3584: 30.7 / 21.6 / 23.8 /
// 21.1; 8192: 66.3 / 45.9 / 49.1 / 41.0 (201 MB: 31 at the copy bandwidth); 592 members of one token 7.6 / 7.4 / 7.9 / 8.3.  (From 1036 to
// 3300 tokens one per CTA is faster by itself, but not in a step: 2048 tokens of 28 / 4 heads 90.9 us with one, 89.2 with four.)
// fp32, one token with two CTAs on an SM and two tokens: 256 tokens 5.3 / 5.3; 360: 8.1 / 6.1; 512: 8.9 / 7.0; 1024: 15.4 / 12.1; 8192: 95 / 70.5.
template <typename T>
static cudaError_t launch_type(const RopeAppendArgs &a, bool interleaved, int batch, cudaStream_t s) {
    const int64_t tokens = (int64_t)a.n * batch, sms = a.sms;
    if (tokens <= 2 * sms) return launch_tok<T, 1, 2>(a, interleaved, batch, s);
    if constexpr (sizeof(T) == 4) return launch_tok<T, 2, 2>(a, interleaved, batch, s);      // (no batches of fp32 caches)
    else return tokens < 7 * sms || a.n < 4 ? launch_tok<T, 1, 4>(a, interleaved, batch, s) : launch_tok<T, 4, 2>(a, interleaved, batch, s);
}

cudaError_t launch_rope_append(const RopeAppendArgs &a, int dtype, bool interleaved, int batch, cudaStream_t s) {
    return dtype == 0 ? launch_type<__nv_bfloat16>(a, interleaved, batch, s) : launch_type<float>(a, interleaved, batch, s);
}

}  // namespace kvf
