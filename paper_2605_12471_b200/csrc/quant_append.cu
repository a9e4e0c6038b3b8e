// Quantised cache storage: rotate + quantise + append.
//
// The paper's Discussion perturbs the stored K/V by a round trip bf16 -> intN -> bf16 and leaves the
// scheme open.  Here a stored row (one token of one KV head, d elements) is symmetric int8 (Q = 127)
// or int4 (Q = 7) with one fp32 scale, decided once when the row is appended:
//     amax = max |x_j|     inv = Q / amax       scale = amax / Q          (fp32, round to nearest)
//     code_j = clamp(rint(x_j * inv), -Q, Q)                               (ties to even)
//     value seen by the attention = bf16(code_j * scale)                   (fp32 product, one rounding;
//                                   code_j * scale itself in the decode kernel, attn_q8_decode.cu)
// For a key row x is the rotated row in fp32 (same operation order as the bf16 path, before any
// rounding to bf16); a value row is quantised as given.  amax = 0 gives codes 0 and scale 0.
// The cache then holds d + 4 (int8) or d / 2 + 4 (int4: code + 8, two to a byte, element 2i in the low
// nibble of byte i) bytes per row instead of 2 d; the attention kernel for long chunks expands code tiles to
// bf16 tiles in shared memory.  Paged caches keep codes and scales of 128 tokens of every KV head in one page
// (see QuantPlanes); a batch of paged caches is one launch (blockIdx.y = cache).
#include "kvfold_internal.h"

namespace kvf {
namespace {

constexpr int kThreads = 512;  // 16 warps: a warp has three of a Llama-shaped token's 48 rows (each a load, a warp reduction and a store)

__device__ __forceinline__ float bf16_lo(uint32_t w) { return __uint_as_float(w << 16); }
__device__ __forceinline__ float bf16_hi(uint32_t w) { return __uint_as_float(w & 0xFFFF0000u); }

__device__ __forceinline__ void rotate(float a, float b, float c, float s, float &ra, float &rb) {
    float cross_a = __fmul_rn(b, s);
    float cross_b = __fmul_rn(a, s);
    ra = __fmaf_rn(a, c, -cross_a);
    rb = __fmaf_rn(b, c, cross_b);
}

// codes of four values of a row held by one lane; the row's scale comes back in `scale`
template <int BITS>
__device__ __forceinline__ void quantise4(const float (&x)[4], int (&code)[4], float &scale) {
    constexpr float Q = BITS == 4 ? 7.f : 127.f;
    float amax = fmaxf(fmaxf(fabsf(x[0]), fabsf(x[1])), fmaxf(fabsf(x[2]), fabsf(x[3])));
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, o));
    const float inv = amax > 0.f ? __fdiv_rn(Q, amax) : 0.f;
    scale = __fdiv_rn(amax, Q);
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        float r = rintf(__fmul_rn(x[e], inv));
        r = fminf(fmaxf(r, -Q), Q);
        code[e] = (int)r;
    }
}

// One warp per row (d = 128: four elements per lane).  Query rows are rotated and written as bf16;
// key rows are rotated in fp32, quantised and appended; value rows are quantised and appended.
// kTok = tokens per CTA, kResident = CTAs of an SM (see launch_bits); a warp takes the same rows of every token, so that up to four tokens' loads
// and reductions are in flight together.
template <bool INTERLEAVED, int BITS, int kTok, int kResident>
__global__ void __launch_bounds__(kThreads, kResident) rope_append_q8_kernel(const RopeAppendArgs a, const QuantPlanes qp) {
    constexpr int RB = 128 * BITS / 8;          // bytes of a stored row
    __shared__ float2 cs[kTok][kMaxHalfDim];   // (cos, sin) per (token, pair)
    constexpr int d = 128, half = 64;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int tok0 = blockIdx.x * kTok;
    const int b = blockIdx.y;      // cache of a batch (0 when there is one cache)

    pdl_launch_dependents();
    // (the per-cache arrays of a ragged batch were written by an earlier kernel of the stream: under
    // a dependent launch they are visible only after the wait)
    if (a.prefixes || a.pos0s) pdl_wait();
    const int64_t prefix = a.prefixes ? a.prefixes[b] : a.prefix;
    const int64_t pos0 = a.pos0s ? a.pos0s[b] : a.pos0;
    const int n = a.ns ? (int)a.ns[b] : a.n;               // tokens this cache folds (a.n: the longest chunk, the stride)
    const int ntok = max(0, min(kTok, n - tok0));
    const int32_t *page_table = a.page_tables ? a.page_tables[b] : a.page_table;
    // where row `row` of KV head g lives: byte offset of its codes from the code block, index of its scale
    auto code_off = [&](int g, int64_t row) -> int64_t {
        if (qp.page_bytes == 0) return ((int64_t)g * a.capacity + row) * RB;
        return (int64_t)page_table[row / kKvTile] * qp.page_bytes + ((int64_t)g * kKvTile + row % kKvTile) * RB;
    };
    auto scale_idx = [&](int g, int64_t row) -> int64_t {
        if (qp.page_bytes == 0) return (int64_t)g * qp.scale_stride + row;
        return (int64_t)page_table[row / kKvTile] * (qp.page_bytes / 4) + (int64_t)g * kKvTile + row % kKvTile;
    };
    for (int idx = threadIdx.x; idx < ntok * half; idx += kThreads) {
        int t = idx / half, j = idx % half;
        double theta = (double)(pos0 + tok0 + t) * a.table.inv_freq[j];
        double sn, cn;
        sincos(theta, &sn, &cn);
        cs[t][j] = make_float2((float)cn, (float)sn);
    }
    const int64_t qoff = (int64_t)b * a.n * a.H * d, koff = (int64_t)b * a.n * a.Hkv * d;
    const __nv_bfloat16 *q = reinterpret_cast<const __nv_bfloat16 *>(a.q) + qoff;
    const __nv_bfloat16 *k = reinterpret_cast<const __nv_bfloat16 *>(a.k_new) + koff;
    const __nv_bfloat16 *v = reinterpret_cast<const __nv_bfloat16 *>(a.v_new) + koff;
    __nv_bfloat16 *qr = reinterpret_cast<__nv_bfloat16 *>(a.q_rot) + qoff;
    const int heads = a.H + (a.k_new ? 2 * a.Hkv : 0);     // query rows, key rows, value rows (queries only: kvf_attend)
    // (the inputs' lines are called into L2 while the kernel before still finishes, as in rope_append.cu: two lines to a row, a warp's
    // first four rows)
    if (lane < 8) {
        const int hh = warp + (lane >> 1) * (kThreads / 32);
        const bool is_q = hh < a.H, is_v = hh >= a.H + a.Hkv;
        const int g = is_q ? hh : is_v ? hh - a.H - a.Hkv : hh - a.H, row_heads = is_q ? a.H : a.Hkv;
        const __nv_bfloat16 *row = (is_q ? q : is_v ? v : k) + ((int64_t)tok0 * row_heads + g) * d + (lane & 1) * half;
#pragma unroll
        for (int u = 0; u < kTok; ++u)
            if (hh < heads && u < ntok) asm volatile("prefetch.global.L2 [%0];" ::"l"(row + (int64_t)u * row_heads * d));
    }
    __syncthreads();
    pdl_wait();   // the table above needs nothing from earlier kernels; the writes below do

    // Rows between the new end of the cache and the next key-tile boundary get value scale 0: the
    // attention expands them to zeros whatever their codes are, so a zero probability never
    // multiplies non-finite bits.
    if (blockIdx.x == 0 && n > 0 && a.k_new) {
        const int zero_rows = a.prefixes ? (int)((kKvTile - (prefix + n) % kKvTile) % kKvTile) : a.zero_rows;
        for (int i = threadIdx.x; i < zero_rows * a.Hkv; i += kThreads)
            qp.v_scales[scale_idx(i / zero_rows, prefix + n + i % zero_rows)] = 0.f;
    }

    for (int hh = warp; hh < heads; hh += kThreads / 32) {
        const bool is_q = hh < a.H, is_v = hh >= a.H + a.Hkv;
        const int g = is_q ? hh : is_v ? hh - a.H - a.Hkv : hh - a.H;        // query head, or KV head
        const int row_heads = is_q ? a.H : a.Hkv;
        const __nv_bfloat16 *src = (is_q ? q : is_v ? v : k) + ((int64_t)tok0 * row_heads + g) * d;
        // where my four elements sit in the row: x[0..1] at e0, x[2..3] at e1.  Value rows and interleaved pairs: 4 lane
        // .. 4 lane + 3; else the pairs (j, j + 64) for j = 2 lane, 2 lane + 1
        const bool in_order = INTERLEAVED || is_v;
        const int e0 = in_order ? 4 * lane : 2 * lane, e1 = in_order ? 4 * lane + 2 : half + 2 * lane;
        // (Rows in order are loaded and stored in two pieces as well: one piece behind a branch of the warp took as long, 2048
        // tokens 20.5 / 20.7 us.)
        // (one turn; without the loop the compiler's order costs two and four tokens 2 - 4 % of a launch)
#pragma unroll 1
        for (int t0 = 0; t0 < ntok; t0 += kTok) {
            uint32_t w0[kTok], w1[kTok];
#pragma unroll
            for (int u = 0; u < kTok; ++u) {
                w0[u] = w1[u] = 0u;
                if (t0 + u < ntok) {
                    const __nv_bfloat16 *p = src + (int64_t)(t0 + u) * row_heads * d;
                    w0[u] = *reinterpret_cast<const uint32_t *>(p + e0);
                    w1[u] = *reinterpret_cast<const uint32_t *>(p + e1);
                }
            }
#pragma unroll
            for (int u = 0; u < kTok; ++u) {
                const int t = t0 + u;
                if (t >= ntok) break;
                const int64_t tok = tok0 + t, cache_row = prefix + tok;
                float x[4];
                if (is_v) {
                    x[0] = bf16_lo(w0[u]); x[1] = bf16_hi(w0[u]); x[2] = bf16_lo(w1[u]); x[3] = bf16_hi(w1[u]);
                } else {
                    const float2 c0 = cs[t][2 * lane], c1 = cs[t][2 * lane + 1];
                    if (!INTERLEAVED) {
                        rotate(bf16_lo(w0[u]), bf16_lo(w1[u]), c0.x, c0.y, x[0], x[2]);
                        rotate(bf16_hi(w0[u]), bf16_hi(w1[u]), c1.x, c1.y, x[1], x[3]);
                    } else {
                        rotate(bf16_lo(w0[u]), bf16_hi(w0[u]), c0.x, c0.y, x[0], x[1]);
                        rotate(bf16_lo(w1[u]), bf16_hi(w1[u]), c1.x, c1.y, x[2], x[3]);
                    }
                }
                if (is_q) {
                    __nv_bfloat16 *dst = qr + (tok * a.H + g) * d;
                    *reinterpret_cast<__nv_bfloat162 *>(dst + e0) = __floats2bfloat162_rn(x[0], x[1]);
                    *reinterpret_cast<__nv_bfloat162 *>(dst + e1) = __floats2bfloat162_rn(x[2], x[3]);
                    continue;
                }
                int code[4];
                float scale;
                quantise4<BITS>(x, code, scale);
                int8_t *codes = (is_v ? qp.v_codes : qp.k_codes) + code_off(g, cache_row);
                if (BITS == 8) {
                    *reinterpret_cast<uint16_t *>(codes + e0) = (uint16_t)((code[0] & 0xFF) | ((code[1] & 0xFF) << 8));
                    *reinterpret_cast<uint16_t *>(codes + e1) = (uint16_t)((code[2] & 0xFF) | ((code[3] & 0xFF) << 8));
                } else {
                    // elements e0, e0 + 1 share byte e0 / 2 (e0 and e1 are even)
                    codes[e0 / 2] = (int8_t)((code[0] + 8) | ((code[1] + 8) << 4));
                    codes[e1 / 2] = (int8_t)((code[2] + 8) | ((code[3] + 8) << 4));
                }
                if (lane == 0) (is_v ? qp.v_scales : qp.k_scales)[scale_idx(g, cache_row)] = scale;
            }
        }
    }
}

template <int BITS, int TOK, int RESIDENT>
cudaError_t launch_tok(const RopeAppendArgs &a, const QuantPlanes &qp, bool interleaved, int batch, cudaStream_t s) {
    auto kernel = interleaved ? rope_append_q8_kernel<true, BITS, TOK, RESIDENT> : rope_append_q8_kernel<false, BITS, TOK, RESIDENT>;
    return launch_pdl(kernel, dim3((a.n + TOK - 1) / TOK, batch), dim3(kThreads), 0, s, a, qp);
}

// As for bf16 rows (rope_append.cu): one token per CTA while two CTAs on an SM hold the launch, and where the members of a batch
// have one each (then four on an SM: 32 registers); else two tokens, from six tokens an SM on four.  us per launch, cold inputs, plain
// launches back to back, int8, 32 / 8 heads, one token with two / four CTAs on an SM, two, four tokens: 256 tokens 5.1 / 5.5 / 5.8 / 8.0; 360:
// 8.6 / 6.7 / 6.5 / 8.1; 512: 9.1 / 8.1 / 6.7 / 8.3; 640: 11.9 / 9.9 / 10.4 / 10.0; 900: 15.0 / 12.1 / 11.7 / 10.3; 2048: 28.0 / 22.3 / 21.7 / 19.7;
// 8192: 104 / 79 / 75 / 64; members of one token, 297: 7.7 / 7.3 / 8.2 / 9.1; 360 of 28 / 4 heads: 8.2 / 7.3 / 8.9 / 9.9; 1024: 17.4 / 18.1 /
// 18.3 / 20.0.
template <int BITS>
cudaError_t launch_bits(const RopeAppendArgs &a, const QuantPlanes &qp, bool interleaved, int batch, cudaStream_t s) {
    const int64_t tokens = (int64_t)a.n * batch, sms = a.sms;
    if (tokens <= 2 * sms) return launch_tok<BITS, 1, 2>(a, qp, interleaved, batch, s);
    if (a.n < 2) return launch_tok<BITS, 1, 4>(a, qp, interleaved, batch, s);
    return tokens < 6 * sms || a.n < 4 ? launch_tok<BITS, 2, 2>(a, qp, interleaved, batch, s) : launch_tok<BITS, 4, 2>(a, qp, interleaved, batch, s);
}

}  // namespace

cudaError_t launch_rope_append_q8(const RopeAppendArgs &a, const QuantPlanes &qp, bool interleaved, int batch, cudaStream_t s) {
    return qp.bits == 4 ? launch_bits<4>(a, qp, interleaved, batch, s) : launch_bits<8>(a, qp, interleaved, batch, s);
}

}  // namespace kvf
