// A whole small fold step in one launch (head_dim 64, CUDA cores): rotate, append, attention, merge.
//
// The steps of a small model are a few microseconds of arithmetic behind three dependent launches (rotate +
// append, attention, merge), and the attention kernel of attn_simt.cu, built for long key ranges, gives 256 query
// rows to four to eight CTAs that walk their key tiles one after the other.  Here a CTA owns 32 query rows
// (row = token * G + head-in-group) and one of up to 16 slices of the key tiles; the CTAs of a row tile form a
// cluster and merge their (maximum, sum, output) through distributed shared memory, each finishing its share of
// the rows.  A CTA rotates its own query rows, and the chunk's own keys where its slice holds them (no CTA reads
// what another one writes); the CTAs of the last row tile, whose slices cover every row of the chunk, also write the
// rotated keys and the values to the cache.  The tables of cosines and sines are worked out before the dependent
// launch's wait, under the tail of the step before.  Arithmetic as in rope_append.cu (the cache bits are a
// contract) and attn_simt.cu (fp32 throughout).
//
// Section 2 of the paper: positions continue from the chunk's absolute start, rows of earlier chunks are all
// visible, rows of the chunk causally.
//
// Measured (fp32, 64 tokens of 4 / 1 heads at prefix 448, replayed back to back): 33.9 us per step through the three
// kernels, 7.1 us here, 5.0 at prefix 0 (launch, one trip to memory, one key tile of 32, the merge).  With the merge as loads
// between two cluster barriers it was 8.7 and 5.6; one token at prefix 500 6.7 -> 4.8.  A key
// tile more in a slice costs 3.7 - 5 us: latency of dependent shared-memory loads at two warps per scheduler (IPC
// 0.34, half of the stall cycles on them), so slices are as short as the device has room for.  Tried: 4 x 4 blocks
// per thread on half the threads (a third less shared-memory traffic, fewer warps: 6.3 us a tile).
#include "kvfold_internal.h"
#include "sm100_ptx.cuh"

namespace kvf {
namespace {

constexpr int BM = 32, kMaxBN = 64, D = 64, HALF = D / 2, kThreads = 256;
constexpr int TR = 2;                // query rows per thread (x BN / 16 keys, x 4 output columns)
constexpr int QS = D + 4;            // padded row stride of the Q, K and probability tiles (floats)
constexpr int kMaxRanks = 1 << (kFoldSmallWidths - 1);     // slices of the key tiles = CTAs of a cluster

struct Smem {
    float q[BM * QS];
    float k[kMaxBN * QS];
    float v[kMaxBN * D];
    float p[BM * QS];
    float2 cs_q[BM][HALF];           // (cos, sin) per (token of the row tile, pair)
    float2 cs_k[kMaxBN][HALF];           // ... per (key of the tile that belongs to the chunk, pair)
    // what the CTAs of the cluster send for this one's BM / ranks rows, by sender: unnormalised outputs, (maximum, sum)
    float landed_o[BM * D];
    float2 landed_ml[BM];
    unsigned long long landed;       // the barrier they complete on
    int abort;
};

__device__ __forceinline__ void unpack(const uint4 &w, float (&x)[4]) {
    x[0] = __uint_as_float(w.x); x[1] = __uint_as_float(w.y); x[2] = __uint_as_float(w.z); x[3] = __uint_as_float(w.w);
}
__device__ __forceinline__ void unpack(const uint4 &w, float (&x)[8]) {
    const uint32_t u[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        x[2 * i] = __uint_as_float(u[i] << 16);
        x[2 * i + 1] = __uint_as_float(u[i] & 0xFFFF0000u);
    }
}
// rounds to the cache's type: the bits for the cache, and the value they stand for in place
__device__ __forceinline__ uint4 pack_round(float (&x)[4]) {
    return make_uint4(__float_as_uint(x[0]), __float_as_uint(x[1]), __float_as_uint(x[2]), __float_as_uint(x[3]));
}
__device__ __forceinline__ uint4 pack_round(float (&x)[8]) {
    uint32_t w[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const uint32_t lo = __bfloat16_as_ushort(__float2bfloat16_rn(x[2 * i])), hi = __bfloat16_as_ushort(__float2bfloat16_rn(x[2 * i + 1]));
        w[i] = lo | (hi << 16);
    }
    const uint4 r = make_uint4(w[0], w[1], w[2], w[3]);
    unpack(r, x);
    return r;
}
__device__ __forceinline__ void rotate(float a, float b, float c, float s, float &ra, float &rb) {
    const float cross_a = __fmul_rn(b, s), cross_b = __fmul_rn(a, s);
    ra = __fmaf_rn(a, c, -cross_a);
    rb = __fmaf_rn(b, c, cross_b);
}
// elements c * N .. of the first half and of the second half of a row, rotated in place
template <int N, bool INTERLEAVED>
__device__ __forceinline__ void rotate_vec(float (&lo)[N], float (&hi)[N], const float2 *cs, int c) {
    if (!INTERLEAVED) {
#pragma unroll
        for (int e = 0; e < N; ++e) {
            const float2 w = cs[c * N + e];
            float a, b;
            rotate(lo[e], hi[e], w.x, w.y, a, b);
            lo[e] = a;
            hi[e] = b;
        }
    } else {
#pragma unroll
        for (int e = 0; e < N; e += 2) {
            const float2 w0 = cs[(c * N + e) / 2], w1 = cs[(HALF + c * N + e) / 2];
            float a, b;
            rotate(lo[e], lo[e + 1], w0.x, w0.y, a, b);
            lo[e] = a; lo[e + 1] = b;
            rotate(hi[e], hi[e + 1], w1.x, w1.y, a, b);
            hi[e] = a; hi[e + 1] = b;
        }
    }
}
template <int N>
__device__ __forceinline__ void to_shared(float *dst, const float (&x)[N]) {
#pragma unroll
    for (int e = 0; e < N; e += 4) *reinterpret_cast<float4 *>(dst + e) = make_float4(x[e], x[e + 1], x[e + 2], x[e + 3]);
}

// BN = keys of a tile: 64, or 32 (see fold_small_cut).
template <typename T, bool INTERLEAVED, int BN>
__global__ void __launch_bounds__(kThreads, 2) fold_small_kernel(const __grid_constant__ RopeAppendArgs r, const __grid_constant__ AttnArgs a) {
    constexpr int VEC = 16 / (int)sizeof(T);
    constexpr int RC = HALF / VEC;                       // vectors of half a row
    constexpr int NK = BN / 16;                          // keys of a thread
    constexpr int KI = (BN * RC + kThreads - 1) / kThreads;               // (first half, second half) vector pairs of a key tile per thread
    constexpr int VI = BN * 2 * RC / kThreads;           // vectors of a value tile per thread
    extern __shared__ __align__(16) uint8_t smem_raw[];
    Smem &sm = *reinterpret_cast<Smem *>(smem_raw);

    const int tid = threadIdx.x, ty = tid >> 4, tx = tid & 15;
    const int tile = blockIdx.x, kvh = blockIdx.y, rank = blockIdx.z, ranks = gridDim.z;
    const int G = a.G, n = a.n;
    const int64_t P = a.prefix;
    const bool writer = r.k_new != nullptr && tile == (int)gridDim.x - 1;

    // this row tile sees the keys below `need`; its key tiles are cut into equal slices
    const int row0 = tile * BM;
    const int tok0 = row0 / G, tok_last = min(n - 1, (row0 + BM - 1) / G);
    const int64_t need = P + (tok_last + 1) * a.self_rows;
    const WindowTiles wt(a.win_lo, a.n_sink, BN);
    const int nt = (int)((need + BN - 1) / BN) - wt.skip;
    const int kt_begin = (int)((int64_t)rank * nt / ranks), kt_end = (int)((int64_t)(rank + 1) * nt / ranks);

    pdl_launch_dependents();
    const uint32_t landed = smem_u32(&sm.landed);
    if (ranks > 1) {
        // (the partners' barriers exist once everybody has been here: waited for ahead of the first store to them)
        if (tid == 0) {
            mbar_init(landed, 1);
            sm.abort = 0;
            asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
            mbar_expect_tx(landed, BM * (D * 4u + 8u));
        }
        __syncwarp();                                     // (.aligned: the warp together)
        cluster_arrive();
    }
    auto table = [&](float2 *cs, int64_t token, int j) {
        const double theta = (double)(r.pos0 + token) * r.table.inv_freq[j];
        double sn, cn;
        sincos(theta, &sn, &cn);
        cs[j] = make_float2((float)cn, (float)sn);
    };
    auto key_table = [&](int kt) {                       // the keys of tile kt that belong to the chunk
        const int64_t key0 = (int64_t)wt.actual(kt) * BN;
        for (int i = tid; i < BN * HALF; i += kThreads) {
            const int64_t key = key0 + i / HALF;
            if (key >= P && key < need) table(sm.cs_k[i / HALF], key - P, i % HALF);
        }
    };
    for (int i = tid; i < (tok_last - tok0 + 1) * HALF; i += kThreads) table(sm.cs_q[i / HALF], tok0 + i / HALF, i % HALF);
    if (kt_begin < kt_end) key_table(kt_begin);
    __syncthreads();
    pdl_wait();      // the tables need nothing from earlier kernels; everything below does

    const T *q = reinterpret_cast<const T *>(r.q);
    const T *k_new = reinterpret_cast<const T *>(r.k_new), *v_new = reinterpret_cast<const T *>(r.v_new);
    T *kp = reinterpret_cast<T *>(r.k_plane) + (int64_t)kvh * r.capacity * D;
    T *vp = reinterpret_cast<T *>(r.v_plane) + (int64_t)kvh * r.capacity * D;
    const uint4 zero = make_uint4(0, 0, 0, 0);

    uint4 klo[KI], khi[KI], vv[VI];
    auto fetch = [&](int kt) {
        const int64_t key0 = (int64_t)wt.actual(kt) * BN;
        auto row_of = [&](const T *plane, const T *fresh, int64_t key) -> const T * {
            if (key >= need) return nullptr;
            return key < P ? plane + key * D : fresh + ((key - P) * r.Hkv + kvh) * D;
        };
#pragma unroll
        for (int u = 0; u < KI; ++u) {
            const int i = tid + u * kThreads;
            if (BN * RC < kThreads && i >= BN * RC) break;
            const T *src = row_of(kp, k_new, key0 + i / RC);
            klo[u] = src ? *reinterpret_cast<const uint4 *>(src + i % RC * VEC) : zero;
            khi[u] = src ? *reinterpret_cast<const uint4 *>(src + HALF + i % RC * VEC) : zero;
        }
#pragma unroll
        for (int u = 0; u < VI; ++u) {
            const int i = tid + u * kThreads;
            const T *src = row_of(vp, v_new, key0 + i / (2 * RC));
            vv[u] = src ? *reinterpret_cast<const uint4 *>(src + i % (2 * RC) * VEC) : zero;
        }
    };
    if (kt_begin < kt_end) fetch(kt_begin);

    // query rows, rotated and rounded to the cache's type as the other kernels read them
    for (int i = tid; i < BM * RC; i += kThreads) {
        const int row = i / RC, c = i % RC, R = row0 + row, tok = R / G, gi = R % G;
        float lo[VEC], hi[VEC];
        const bool valid = tok < n;
        const T *src = q + ((int64_t)tok * a.H + kvh * G + gi) * D;
        unpack(valid ? *reinterpret_cast<const uint4 *>(src + c * VEC) : zero, lo);
        unpack(valid ? *reinterpret_cast<const uint4 *>(src + HALF + c * VEC) : zero, hi);
        if (valid) {
            rotate_vec<VEC, INTERLEAVED>(lo, hi, sm.cs_q[tok - tok0], c);
            pack_round(lo);
            pack_round(hi);
        }
        to_shared(sm.q + row * QS + c * VEC, lo);
        to_shared(sm.q + row * QS + HALF + c * VEC, hi);
    }
    if (writer && r.zero_rows > 0 && rank == ranks - 1) {
        // value rows behind the new end, to the next 128-row boundary (as rope_append.cu leaves them)
        for (int i = tid; i < r.zero_rows * 2 * RC; i += kThreads)
            *reinterpret_cast<uint4 *>(vp + (P + n + i / (2 * RC)) * D + i % (2 * RC) * VEC) = zero;
    }

    int64_t limit[TR];    // keys below limit are visible to row TR * ty + i
#pragma unroll
    for (int i = 0; i < TR; ++i) {
        const int tok = (row0 + TR * ty + i) / G;
        limit[i] = tok < n ? P + (tok + 1) * a.self_rows : 0;
    }
    float m[TR], l[TR];
    float2 acc[TR][2] = {};
#pragma unroll
    for (int i = 0; i < TR; ++i) {
        m[i] = -INFINITY;
        l[i] = 0.f;
    }

    for (int kt = kt_begin; kt < kt_end; ++kt) {
        const int64_t key0 = (int64_t)wt.actual(kt) * BN;
        if (kt > kt_begin) {
            __syncthreads();                              // the tile before has been read
            if (key0 + BN > P) {
                key_table(kt);
                __syncthreads();
            }
        }
#pragma unroll
        for (int u = 0; u < KI; ++u) {
            const int i = tid + u * kThreads, row = i / RC, c = i % RC;
            if (BN * RC < kThreads && i >= BN * RC) break;
            const int64_t key = key0 + row;
            float lo[VEC], hi[VEC];
            unpack(klo[u], lo);
            unpack(khi[u], hi);
            if (key >= P && key < need) {
                rotate_vec<VEC, INTERLEAVED>(lo, hi, sm.cs_k[row], c);
                const uint4 wl = pack_round(lo), wh = pack_round(hi);
                if (writer) {
                    *reinterpret_cast<uint4 *>(kp + key * D + c * VEC) = wl;
                    *reinterpret_cast<uint4 *>(kp + key * D + HALF + c * VEC) = wh;
                }
            }
            to_shared(sm.k + row * QS + c * VEC, lo);
            to_shared(sm.k + row * QS + HALF + c * VEC, hi);
        }
#pragma unroll
        for (int u = 0; u < VI; ++u) {
            const int i = tid + u * kThreads, row = i / (2 * RC), c = i % (2 * RC);
            const int64_t key = key0 + row;
            if (writer && key >= P && key < need) *reinterpret_cast<uint4 *>(vp + key * D + c * VEC) = vv[u];
            float x[VEC];
            unpack(vv[u], x);
            to_shared(sm.v + row * D + c * VEC, x);
        }
        __syncthreads();
        if (kt + 1 < kt_end) fetch(kt + 1);               // in flight under this tile's arithmetic

        // (packed multiply-adds: two sums per score, over even and odd elements)
        float2 s2[TR][NK] = {};
#pragma unroll 4
        for (int k4 = 0; k4 < D / 4; ++k4) {
            float4 qa[TR], kb[NK];
#pragma unroll
            for (int i = 0; i < TR; ++i) qa[i] = *reinterpret_cast<const float4 *>(sm.q + (TR * ty + i) * QS + k4 * 4);
#pragma unroll
            for (int j = 0; j < NK; ++j) kb[j] = *reinterpret_cast<const float4 *>(sm.k + (tx + 16 * j) * QS + k4 * 4);
#pragma unroll
            for (int i = 0; i < TR; ++i)
#pragma unroll
                for (int j = 0; j < NK; ++j) {
                    s2[i][j] = __ffma2_rn(make_float2(qa[i].x, qa[i].y), make_float2(kb[j].x, kb[j].y), s2[i][j]);
                    s2[i][j] = __ffma2_rn(make_float2(qa[i].z, qa[i].w), make_float2(kb[j].z, kb[j].w), s2[i][j]);
                }
        }
        float s[TR][NK];
#pragma unroll
        for (int i = 0; i < TR; ++i) {
            float mx = -INFINITY;
#pragma unroll
            for (int j = 0; j < NK; ++j) {
                const int64_t key = key0 + tx + 16 * j;
                const bool vis = key < limit[i] && (key >= a.win_lo || key < a.n_sink);
                s[i][j] = vis ? (s2[i][j].x + s2[i][j].y) * a.scale_log2 : -INFINITY;
                mx = fmaxf(mx, s[i][j]);
            }
#pragma unroll
            for (int o = 1; o < 16; o <<= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
            const float m_new = fmaxf(m[i], mx), m_safe = m_new == -INFINITY ? 0.f : m_new;
            const float alpha = exp2f(m[i] - m_safe);
            float sum = 0.f;
#pragma unroll
            for (int j = 0; j < NK; ++j) {
                const float p = exp2f(s[i][j] - m_safe);
                sum += p;
                sm.p[(TR * ty + i) * QS + tx + 16 * j] = p;
            }
#pragma unroll
            for (int o = 1; o < 16; o <<= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
            l[i] = l[i] * alpha + sum;
            m[i] = m_new;
#pragma unroll
            for (int c = 0; c < 2; ++c) acc[i][c] = __fmul2_rn(acc[i][c], make_float2(alpha, alpha));
        }
        __syncwarp();                                     // a row's probabilities stay within its half warp
#pragma unroll 4
        for (int k4 = 0; k4 < BN / 4; ++k4) {
            float4 p4[TR];
#pragma unroll
            for (int i = 0; i < TR; ++i) p4[i] = *reinterpret_cast<const float4 *>(sm.p + (TR * ty + i) * QS + k4 * 4);
#pragma unroll
            for (int kk = 0; kk < 4; ++kk) {
                const float4 x = *reinterpret_cast<const float4 *>(sm.v + (k4 * 4 + kk) * D + tx * 4);
#pragma unroll
                for (int i = 0; i < TR; ++i) {
                    const float p = kk == 0 ? p4[i].x : kk == 1 ? p4[i].y : kk == 2 ? p4[i].z : p4[i].w;
                    acc[i][0] = __ffma2_rn(make_float2(p, p), make_float2(x.x, x.y), acc[i][0]);
                    acc[i][1] = __ffma2_rn(make_float2(p, p), make_float2(x.z, x.w), acc[i][1]);
                }
            }
        }
        __syncwarp();                                     // (the next tile's probabilities overwrite these)
    }

    // Every slice's maximum, sum and unnormalised output go to the CTA that finishes the row, which merges them in slice order.
    // (Stores that complete on the receiver's barrier, instead of loads between two cluster barriers.)
    const int rows = BM / ranks;                          // (ranks is a power of two)
    __syncwarp();
    if (ranks > 1) cluster_wait();
#pragma unroll
    for (int i = 0; i < TR; ++i) {
        const int row = TR * ty + i, at = rank * rows + row % rows;
        const float4 o = make_float4(acc[i][0].x, acc[i][0].y, acc[i][1].x, acc[i][1].y);
        if (ranks > 1) {
            const uint32_t to = (uint32_t)(row / rows), done = peer_smem(landed, to);
            peer_store4(peer_smem(smem_u32(&sm.landed_o[at * D + tx * 4]), to), o, done);
            if (tx == 0) peer_store2(peer_smem(smem_u32(&sm.landed_ml[at]), to), make_float2(m[i], l[i]), done);
        } else {
            *reinterpret_cast<float4 *>(&sm.landed_o[at * D + tx * 4]) = o;
            if (tx == 0) sm.landed_ml[at] = make_float2(m[i], l[i]);
        }
    }
    bool ok = true;
    if (ranks == 1) {
        __syncthreads();
    } else {
        __syncwarp();
        cluster_arrive_relaxed();                         // (nothing goes to a partner any more)
        ok = mbar_wait(landed, 0, &sm, a.status);
    }
    for (int i = tid; ok && i < rows * (D / 4); i += kThreads) {
        const int own = i / (D / 4), row = rank * rows + own, c = i % (D / 4);
        const int R = row0 + row, tok = R / G, gi = R % G;
        if (tok >= n) continue;
        float2 ml[kMaxRanks];
        float M = -INFINITY;
#pragma unroll
        for (int s = 0; s < kMaxRanks; ++s) {
            ml[s] = s < ranks ? sm.landed_ml[s * rows + own] : make_float2(-INFINITY, 0.f);
            M = fmaxf(M, ml[s].x);
        }
        const float M0 = M == -INFINITY ? 0.f : M;
        float den = 0.f;
        float4 o = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int s = 0; s < kMaxRanks; ++s) {
            if (s >= ranks) break;
            const float w = exp2f(ml[s].x - M0);
            const float4 x = *reinterpret_cast<const float4 *>(&sm.landed_o[(s * rows + own) * D + c * 4]);
            den = fmaf(w, ml[s].y, den);
            o.x = fmaf(w, x.x, o.x); o.y = fmaf(w, x.y, o.y); o.z = fmaf(w, x.z, o.z); o.w = fmaf(w, x.w, o.w);
        }
        const float inv = den > 0.f ? 1.f / den : 0.f;
        o.x *= inv; o.y *= inv; o.z *= inv; o.w *= inv;
        const int64_t at = (int64_t)tok * a.H + kvh * G + gi;
        if (a.out_f32) {
            *reinterpret_cast<float4 *>(reinterpret_cast<float *>(a.out) + at * D + c * 4) = o;
        } else {
            __nv_bfloat162 b0 = __floats2bfloat162_rn(o.x, o.y), b1 = __floats2bfloat162_rn(o.z, o.w);
            uint2 pk;
            pk.x = *reinterpret_cast<uint32_t *>(&b0);
            pk.y = *reinterpret_cast<uint32_t *>(&b1);
            *reinterpret_cast<uint2 *>(reinterpret_cast<__nv_bfloat16 *>(a.out) + at * D + c * 4) = pk;
        }
        if (c == 0 && a.lse) a.lse[at] = (den > 0.f ? M + log2f(den) : -INFINITY) * 0.6931471805599453f;
    }
    // Nobody leaves while a partner may still store here.  What others send has landed, so they have arrived and this is no wait; where the
    // wait was given up, what they sent before they arrived is waited for: one CTA's time-out must not become a fault of another.
    if (ranks > 1) {
        __syncwarp();
        cluster_wait();
        if (!ok && tid == 0) mbar_wait_drain(landed, 0, a.status);
    }
}

// Once per kernel and device: shared-memory limit, clusters of 16 CTAs (beyond the portable eight), and how many clusters
// of each width the device holds at once.
template <typename T, bool INTERLEAVED, int BN>
cudaError_t prepare_once(FoldSmallFit *fit) {
    struct Done { int dev; FoldSmallFit fit; };
    static std::mutex mu;
    static std::vector<Done> done;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    std::lock_guard<std::mutex> lock(mu);
    for (const Done &d : done)
        if (d.dev == dev) {
            if (fit) *fit = d.fit;
            return cudaSuccess;
        }
    auto kernel = fold_small_kernel<T, INTERLEAVED, BN>;
    e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(Smem));
    if (e != cudaSuccess) return e;
    Done now = {dev, {}};
    const bool wide = cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess;
    bool refused = !wide;
    for (int i = 0; i < kFoldSmallWidths; ++i) {
        if ((1 << i) > 8 && !wide) break;
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(1, 1, 1u << i);
        cfg.blockDim = dim3(kThreads);
        cfg.dynamicSmemBytes = sizeof(Smem);
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = 1;
        attr[0].val.clusterDim.y = 1;
        attr[0].val.clusterDim.z = 1u << i;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        int clusters = 0;
        if (cudaOccupancyMaxActiveClusters(&clusters, kernel, &cfg) == cudaSuccess) now.fit.clusters[i] = clusters;
        else refused = true;
    }
    if (refused) cudaGetLastError();       // (a width the device refuses leaves its error behind)
    done.push_back(now);
    if (fit) *fit = now.fit;
    return cudaSuccess;
}

template <typename T, bool INTERLEAVED, int BN>
cudaError_t launch_bn(const RopeAppendArgs &r, const AttnArgs &a, int ranks, cudaStream_t s) {
    cudaError_t e = prepare_once<T, INTERLEAVED, BN>(nullptr);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(fold_small_row_tiles(a.n, a.G), a.Hkv, ranks);
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = sizeof(Smem);
    cfg.stream = s;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = g_pdl_allowed ? 1 : 0;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = 1;
    attr[1].val.clusterDim.y = 1;
    attr[1].val.clusterDim.z = (unsigned)ranks;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    return cudaLaunchKernelEx(&cfg, fold_small_kernel<T, INTERLEAVED, BN>, r, a);
}

template <typename T, bool INTERLEAVED>
cudaError_t launch_t(const RopeAppendArgs &r, const AttnArgs &a, const FoldSmallCut &cut, cudaStream_t s) {
    return cut.keys == 32 ? launch_bn<T, INTERLEAVED, 32>(r, a, cut.ranks, s) : launch_bn<T, INTERLEAVED, 64>(r, a, cut.ranks, s);
}

}  // namespace

int fold_small_row_tiles(int n, int G) { return (int)(((int64_t)n * G + BM - 1) / BM); }

// Slices of the key tiles = CTAs of a cluster: a power of two, and no more clusters than the device holds at once: a second
// wave costs more than longer slices.  Two CTAs fit an SM, but a cluster stays within one GPC: of 16 CTAs the device holds 14
// clusters (16 row tiles, 24 key tiles: 16 slices 37.4 us, 8 slices 28.6), of 8 CTAs fewer than 36 (36 row tiles, 16 key
// tiles: 8 slices 36.1 us, through three launches 34.4).
int fold_small_ranks(int row_tiles, int64_t key_tiles, const FoldSmallFit &fit) {
    int ranks = 1;
    for (int i = 1; i < kFoldSmallWidths && (1 << i) <= key_tiles && row_tiles <= fit.clusters[i]; ++i) ranks = 1 << i;
    return ranks;
}

// The cut a small step runs with: as many slices as that or more, in tiles of 64 or 32 keys, by what the longest slice costs
// (us per tile: 3.9 while a cluster's CTAs have an SM each, 6.6 where they share it; 32 keys 2.2).  More slices than whole
// tiles fit into (the last ones empty) where that makes the longest one shorter: 64 tokens of 4 / 1 heads, five key tiles in four
// slices 14.5 us, in eight 8.6.  Tiles of 32 keys up to one CTA per SM: 64 tokens at prefix 448 7.55 in eight slices of 64 keys, 7.2 in
// sixteen of 32; 64 tokens of 8 / 2 heads at prefix 700 18.2 / 16.2.  (A window's first tile holds its sinks, up to 64: no tiles of 32.)
FoldSmallCut fold_small_cut(int row_tiles, int64_t keys, bool window, const FoldSmallFit &fit) {
    auto cost = [&](const FoldSmallCut &c) {
        const int64_t tiles = (keys + c.keys - 1) / c.keys, slice = (tiles + c.ranks - 1) / c.ranks;
        const bool alone = 2 * (int64_t)row_tiles * c.ranks <= fit.clusters[0];
        return (double)slice * (c.keys == 32 ? 2.2 : alone ? 3.9 : 6.6) + 0.05 * c.ranks;
    };
    FoldSmallCut best = {64, fold_small_ranks(row_tiles, (keys + 63) / 64, fit)};
    for (int bn = 64; bn >= (window ? 64 : 32); bn -= 32)
        for (int i = 0; i < kFoldSmallWidths; ++i) {
            const FoldSmallCut c = {bn, 1 << i};
            if (row_tiles > fit.clusters[i] || (i > 0 && (int64_t)(c.ranks / 2) * bn >= keys)) break;
            if (bn == 32 && 2 * (int64_t)row_tiles * c.ranks > fit.clusters[0]) break;
            if (c.ranks >= best.ranks && cost(c) < cost(best)) best = c;
        }
    return best;
}

// (the eight kernels differ in arithmetic and tile width only, in neither threads, shared memory nor the limit on registers: what
// fits one fits all)
cudaError_t fold_small_fit(FoldSmallFit *fit) { return prepare_once<float, false, 64>(fit); }

cudaError_t launch_fold_small(const RopeAppendArgs &r, const AttnArgs &a, const FoldSmallCut &cut, int dtype, bool interleaved, cudaStream_t s) {
    if (a.d != D) return cudaErrorInvalidValue;
    if (dtype == 0) return interleaved ? launch_t<__nv_bfloat16, true>(r, a, cut, s) : launch_t<__nv_bfloat16, false>(r, a, cut, s);
    return interleaved ? launch_t<float, true>(r, a, cut, s) : launch_t<float, false>(r, a, cut, s);
}

}  // namespace kvf
