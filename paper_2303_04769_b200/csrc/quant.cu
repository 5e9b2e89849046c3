// Quantised inference (paper Sections 5.1 and 5.5: uint8 tensors; Section 5.3: int32 accumulation) over the same
// blocked layout with one byte per channel: uint8[N][ceil(C/32)][H][W][32], a pixel of a channel block = 32 bytes = 8
// words of 4 channels; pad lanes hold 0.  This file: the layout moves, the filter packing, the bandwidth-bound layers
// (depthwise, max pool, ReLU) and the C ABI of the quantised layers; the full channel reduction runs on the tensor cores
// (conv_i8.cu).  Arithmetic: acc = bias + sum (q_in - z_in)(q_w - z_w) in int32,
// q_out = clamp(z_out + floor((acc * mult + 2^(shift-1)) / 2^shift), lo, 255) with a 64-bit product, lo = z_out under
// ReLU.  Max pooling and ReLU act on the bytes themselves (the affine map keeps order).
#include "common.cuh"

namespace small {

namespace {

__device__ __forceinline__ int requantize(int acc, int mult, int shift, int zo, int lo) {
    const long long r = ((long long)acc * (long long)mult + (1ll << (shift - 1))) >> shift;
    const long long z = (long long)zo + r;
    return (int)(z < lo ? lo : z > 255 ? 255 : z);
}

// one thread = one word (4 channels) of one pixel of the blocked tensor
__global__ void q_pack_kernel(const uint8_t *__restrict__ nchw, uint32_t *__restrict__ blk, int C, int HW, int CB, size_t words) {
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < words; i += (size_t)gridDim.x * blockDim.x) {
        const int c4 = (int)(i & 7);
        size_t r = i >> 3;
        const int p = (int)(r % HW); r /= HW;
        const int cb = (int)(r % CB);
        const size_t n = r / CB;
        uint32_t word = 0;
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            const int c = cb * 32 + c4 * 4 + b;
            if (c < C) word |= (uint32_t)nchw[(n * C + c) * HW + p] << (8 * b);
        }
        blk[i] = word;
    }
}

__global__ void q_unpack_kernel(const uint32_t *__restrict__ blk, uint8_t *__restrict__ nchw, int C, int HW, int CB, size_t words) {
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < words; i += (size_t)gridDim.x * blockDim.x) {
        const int c4 = (int)(i & 7);
        size_t r = i >> 3;
        const int p = (int)(r % HW); r /= HW;
        const int cb = (int)(r % CB);
        const size_t n = r / CB;
        const uint32_t word = blk[i];
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            const int c = cb * 32 + c4 * 4 + b;
            if (c < C) nchw[(n * C + c) * HW + p] = (uint8_t)(word >> (8 * b));
        }
    }
}

// filters [K][C][FH][FW] bytes -> [CB][T][KB * 32 filters][32 channels]: 32 bytes of a filter, tap and channel block are one
// K step of the tensor core's byte MMA (conv_i8.cu), stored in the order of the 32-byte swizzle so that a box of filters is one
// contiguous copy; pad channels and pad filters 0
__global__ void pack_q_conv_w_kernel(const uint8_t *__restrict__ w, uint32_t *__restrict__ wb, int C, int K, int T, size_t words) {
    const int Kp = (K + 31) / 32 * 32;
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < words; i += (size_t)gridDim.x * blockDim.x) {
        size_t r = i;
        const int k = (int)((r >> 3) % Kp);
        const int c4 = (int)(r & 7) ^ (k & 4);      // rows 4-7 of every 8 hold their two 16-byte halves exchanged
        r = (r >> 3) / Kp;
        const int t = (int)(r % T);
        const int cb = (int)(r / T);
        uint32_t word = 0;
        if (k < K)
#pragma unroll
            for (int b = 0; b < 4; ++b) {
                const int c = cb * 32 + c4 * 4 + b;
                if (c < C) word |= (uint32_t)w[((size_t)k * C + c) * T + t] << (8 * b);
            }
        wb[i] = word;
    }
}

// per filter and tap the sum of the weight bytes over the channels [K][T]
__global__ void q_conv_tables_kernel(const uint8_t *__restrict__ w, int *__restrict__ tab, int C, int K, int T) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= K * T) return;
    const int k = i / T, t = i - k * T;
    int s = 0;
    for (int c = 0; c < C; ++c) s += w[((size_t)k * C + c) * T + t];
    tab[i] = s;
}

// depthwise filters [C][FH][FW] bytes -> [CB][T][32] bytes, pad lanes 0
__global__ void pack_q_dw_w_kernel(const uint8_t *__restrict__ w, uint8_t *__restrict__ wb, int C, int T, int total) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= total) return;
    const int lane = i & 31, t = (i >> 5) % T, cb = (i >> 5) / T;
    const int c = cb * 32 + lane;
    wb[i] = c < C ? w[(size_t)c * T + t] : (uint8_t)0;
}

struct QPlaneArgs {
    const uint32_t *in; uint32_t *out; const uint32_t *w; const int *bias;
    int N, C, CB, H, W, FH, FW, S, pt, pl, OH, OW;
    int zx, zw, zo, mult, shift, lo;
};

// one thread = 4 channels of one output pixel; any window, stride and padding
__global__ void q_dwconv_kernel(const QPlaneArgs a) {
    const size_t words = (size_t)a.N * a.CB * a.OH * a.OW * 8;
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < words; i += (size_t)gridDim.x * blockDim.x) {
        const int c4 = (int)(i & 7);
        size_t r = i >> 3;
        const int ow = (int)(r % a.OW); r /= a.OW;
        const int oh = (int)(r % a.OH); r /= a.OH;
        const int cb = (int)(r % a.CB);
        const size_t n = r / a.CB;
        const uint32_t *plane = a.in + ((n * a.CB + cb) * a.H * a.W) * 8 + c4;
        int acc[4] = {0, 0, 0, 0};
        for (int x = 0; x < a.FH; ++x) {
            const int ih = oh * a.S + x - a.pt;
            if (ih < 0 || ih >= a.H) continue;
            for (int y = 0; y < a.FW; ++y) {
                const int iw = ow * a.S + y - a.pl;
                if (iw < 0 || iw >= a.W) continue;
                const uint32_t xv = plane[((size_t)ih * a.W + iw) * 8];
                const uint32_t wv = a.w[((size_t)cb * a.FH * a.FW + x * a.FW + y) * 8 + c4];
#pragma unroll
                for (int b = 0; b < 4; ++b)
                    acc[b] += ((int)((xv >> (8 * b)) & 255u) - a.zx) * ((int)((wv >> (8 * b)) & 255u) - a.zw);
            }
        }
        uint32_t word = 0;
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            const int c = cb * 32 + c4 * 4 + b;
            if (c < a.C) word |= (uint32_t)requantize(acc[b] + (a.bias ? a.bias[c] : 0), a.mult, a.shift, a.zo, a.lo) << (8 * b);
        }
        a.out[i] = word;
    }
}

__device__ __forceinline__ uint32_t lane_mask(int C, int cb, int c4) {      // 0xff in the bytes of real channels
    uint32_t m = 0;
#pragma unroll
    for (int b = 0; b < 4; ++b)
        if (cb * 32 + c4 * 4 + b < C) m |= 0xffu << (8 * b);
    return m;
}

__device__ __forceinline__ uint64_t pair(float x, float y) {
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(x), "f"(y));
    return r;
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
    uint64_t r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) {
    uint64_t r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
// Requantisation of an int32 sum as one 64-bit multiply-add: everything that does not depend on the sum is in the addend.
// For 32 <= shift <= 43 (FAST) that includes the output's zero point << shift - |sum + bias| * mult, the rounding half and
// it stay below 2^63 there, as |sum| <= 33000 * 255^2 - and the high word alone is shifted.
__device__ __forceinline__ long long requant_addend(int bias, int mult, int shift, int zo) {
    return (long long)bias * mult + (1ll << (shift - 1)) + ((long long)zo << shift);
}
__device__ __forceinline__ uint32_t requant4_fast(const int (&v)[4], int mult, const long long (&add)[4], int sh, int lo) {
    int q[4];
#pragma unroll
    for (int b = 0; b < 4; ++b) q[b] = max((int)(((long long)v[b] * (long long)mult + add[b]) >> 32) >> sh, lo);
    uint32_t l, h;                                 // two values saturated to bytes each
    asm("cvt.pack.sat.u8.s32.b32 %0, %1, %2, %3;" : "=r"(l) : "r"(q[1]), "r"(q[0]), "r"(0u));
    asm("cvt.pack.sat.u8.s32.b32 %0, %1, %2, %3;" : "=r"(h) : "r"(q[3]), "r"(q[2]), "r"(0u));
    return __byte_perm(l, h, 0x5410);
}
__device__ __forceinline__ uint32_t requant4(const int (&v)[4], int mult, const long long (&add)[4], int shift, int zo, int lo) {
    uint32_t w = 0;
#pragma unroll
    for (int b = 0; b < 4; ++b) {
        const long long r = (((long long)v[b] * (long long)mult + add[b]) >> shift) + zo;
        w |= (uint32_t)(r < lo ? lo : r > 255 ? 255 : (int)r) << (8 * b);
    }
    return w;
}
// bytes b and b + 1 of a word as floats minus a zero point: a byte under the exponent of 2^23 is 2^23 + its value, and `sub`
// holds -(2^23 + zero point) twice
template <int B>
__device__ __forceinline__ uint64_t bytes_f2(uint32_t word, uint64_t sub) {
    return add2(pair(__uint_as_float(__byte_perm(word, 0x4b000000u, 0x7440 | B)), __uint_as_float(__byte_perm(word, 0x4b000000u, 0x7440 | (B + 1)))), sub);
}

// 3 x 3 windows, strides 1 and 2.  Bounded by instructions, not by its bytes (a quarter of the float layer's).  The sums are
// below 9 * 255^2 < 2^24, so single-precision FMAs compute them exactly, two channels per instruction (f32x2).  A thread
// walks down a run of output rows of its column: every input row is converted once and added to the two or three outputs
// whose window it is in, and the next rows' words are in flight meanwhile.  Measured at 512 x 64 channels x 25 x 5: 8.9 us
// (one output per thread 17.3: unpacking the filters and dividing the index cost more than the window; bytewise integer
// multiply-adds before that 70).  Pixels outside the plane are the zero point, which is a real zero.
// FAST: 32 <= shift <= 43 (see requant_addend).
template <int S, bool FAST>
__global__ void __launch_bounds__(128, 5) q_dw3x3_kernel(const QPlaneArgs a, int R, unsigned segs, unsigned items) {
    constexpr int kRing = S == 1 ? 3 : 2;          // outputs whose windows overlap an input row's
    constexpr int U = S == 1 ? 3 : 4;              // input rows per trip: a multiple of the ring's period
    const unsigned i = blockIdx.x * 128u + threadIdx.x;
    grid_dep_sync();
    grid_dep_trigger();
    if (i >= items) return;
    const int c4 = (int)(i & 7u);
    unsigned r = i >> 3;
    const int ow = (int)(r % (unsigned)a.OW); r /= (unsigned)a.OW;
    const int seg = (int)(r % segs);
    const unsigned plane = r / segs;
    const int cb = (int)(plane % (unsigned)a.CB);
    const int oh0 = seg * R, ih0 = oh0 * S - a.pt, iw = ow * S - a.pl;
    const int n_in = (min(R, a.OH - oh0) - 1) * S + 3;
    const uint32_t *src = a.in + ((ptrdiff_t)plane * a.H * a.W + (ptrdiff_t)ih0 * a.W + iw) * 8 + c4;
    const uint32_t z4 = (uint32_t)a.zx * 0x01010101u;
    bool col[3];
#pragma unroll
    for (int y = 0; y < 3; ++y) col[y] = (unsigned)(iw + y) < (unsigned)a.W;
    const int pitch = a.W * 8;
    int k_next = 0;                                // rows are loaded in order
    const int k_lo = max(0, -ih0), k_hi = min(n_in, a.H - ih0);
    auto load = [&](uint32_t (&x)[3]) {
        const bool row = k_next >= k_lo && k_next < k_hi;
#pragma unroll
        for (int y = 0; y < 3; ++y) x[y] = row && col[y] ? src[y * 8] : z4;
        src += pitch;
        ++k_next;
    };
    uint32_t x[U][3], wr[9];
#pragma unroll
    for (int u = 0; u < U; ++u) load(x[u]);
#pragma unroll
    for (int k = 0; k < 9; ++k) wr[k] = a.w[(cb * 9 + k) * 8 + c4];
    long long add[4];                              // bias * mult + the rounding half
#pragma unroll
    for (int b = 0; b < 4; ++b)
        add[b] = requant_addend(a.bias && cb * 32 + c4 * 4 + b < a.C ? a.bias[cb * 32 + c4 * 4 + b] : 0, a.mult, a.shift, FAST ? a.zo : 0) -
                 0x4b400000ll * a.mult;
    const float fx = -(8388608.0f + (float)a.zx), fw = -(8388608.0f + (float)a.zw);
    const uint64_t sub_x = pair(fx, fx), sub_w = pair(fw, fw), start = pair(12582912.0f, 12582912.0f);     // 1.5 * 2^23: the sum's integer in the low bits
    uint64_t w[9][2], acc[kRing][2];
#pragma unroll
    for (int k = 0; k < 9; ++k) { w[k][0] = bytes_f2<0>(wr[k], sub_w); w[k][1] = bytes_f2<2>(wr[k], sub_w); }
#pragma unroll
    for (int o = 0; o < kRing; ++o) acc[o][0] = acc[o][1] = start;
    const uint32_t lanes = lane_mask(a.C, cb, c4);
    uint32_t *dst = a.out + (((size_t)plane * a.OH + oh0) * a.OW + ow) * 8 + c4;
    for (int k0 = 0; k0 < n_in; k0 += U) {
        uint32_t nx[U][3];
#pragma unroll
        for (int u = 0; u < U; ++u) load(nx[u]);
#pragma unroll
        for (int u = 0; u < U; ++u) {              // input row k0 + u is row t of the window of output (k0 + u - t) / S
#pragma unroll
            for (int y = 0; y < 3; ++y) {
                const uint64_t v0 = bytes_f2<0>(x[u][y], sub_x), v1 = bytes_f2<2>(x[u][y], sub_x);
#pragma unroll
                for (int t = 0; t < 3; ++t) {
                    if ((u + 2 * S - t) % S != 0) continue;
                    const int o = ((u + U * S - t) / S) % kRing;
                    acc[o][0] = fma2(v0, w[t * 3 + y][0], acc[o][0]);
                    acc[o][1] = fma2(v1, w[t * 3 + y][1], acc[o][1]);
                }
            }
            if (u % S == 0) {                      // its last row: output (k0 + u - 2) / S is complete
                const int k = k0 + u, o = ((u + U * S - 2) / S) % kRing;
                if (k >= 2 && k < n_in) {
                    const int v[4] = {(int)(uint32_t)acc[o][0], (int)(acc[o][0] >> 32), (int)(uint32_t)acc[o][1], (int)(acc[o][1] >> 32)};
                    *dst = (FAST ? requant4_fast(v, a.mult, add, a.shift - 32, a.lo) : requant4(v, a.mult, add, a.shift, a.zo, a.lo)) & lanes;
                    dst += (size_t)a.OW * 8;
                }
                acc[o][0] = acc[o][1] = start;
            }
        }
#pragma unroll
        for (int u = 0; u < U; ++u)
#pragma unroll
            for (int y = 0; y < 3; ++y) x[u][y] = nx[u][y];
    }
}

// one thread = 16 channels of one output pixel (IndexT: 32 bits where they hold the item count - a 64-bit division costs
// more than the whole window)
template <typename IndexT>
__global__ void __launch_bounds__(256) q_maxpool_kernel(const QPlaneArgs a, IndexT items) {
    const uint32_t z4 = (uint32_t)a.zx * 0x01010101u;
    grid_dep_sync();
    grid_dep_trigger();
    for (IndexT i = blockIdx.x * (IndexT)256 + threadIdx.x; i < items; i += (IndexT)gridDim.x * 256) {
        const int half = (int)(i & 1);
        IndexT r = i >> 1;
        const int ow = (int)(r % (IndexT)a.OW); r /= (IndexT)a.OW;
        const int oh = (int)(r % (IndexT)a.OH);
        const IndexT plane = r / (IndexT)a.OH;
        const int cb = (int)(plane % (IndexT)a.CB);
        const uint4 *src = reinterpret_cast<const uint4 *>(a.in) + (size_t)plane * a.H * a.W * 2 + half;
        const int ih0 = oh * a.S - a.pt, iw0 = ow * a.S - a.pl;
        const int x0 = max(0, -ih0), x1 = min(a.FH, a.H - ih0), y0 = max(0, -iw0), y1 = min(a.FW, a.W - iw0);
        uint4 best = x0 < x1 && y0 < y1 ? make_uint4(0u, 0u, 0u, 0u) : make_uint4(z4, z4, z4, z4);
        for (int x = x0; x < x1; ++x)
            for (int y = y0; y < y1; ++y) {
                const uint4 v = src[((size_t)(ih0 + x) * a.W + iw0 + y) * 2];
                best.x = __vmaxu4(best.x, v.x); best.y = __vmaxu4(best.y, v.y); best.z = __vmaxu4(best.z, v.z); best.w = __vmaxu4(best.w, v.w);
            }
        const int c4 = half * 4;
        best.x &= lane_mask(a.C, cb, c4); best.y &= lane_mask(a.C, cb, c4 + 1); best.z &= lane_mask(a.C, cb, c4 + 2); best.w &= lane_mask(a.C, cb, c4 + 3);
        reinterpret_cast<uint4 *>(a.out)[i] = best;
    }
}

__global__ void q_relu_kernel(const uint32_t *__restrict__ in, uint32_t *__restrict__ out, int C, int CB, int HW, int z, size_t words) {
    const uint32_t z4 = (uint32_t)z * 0x01010101u;
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < words; i += (size_t)gridDim.x * blockDim.x) {
        const int c4 = (int)(i & 7);
        const int cb = (int)((i >> 3) / HW % CB);
        out[i] = __vmaxu4(in[i], z4) & lane_mask(C, cb, c4);
    }
}

int grid_for(small_ctx *ctx, size_t items) {
    const size_t want = (items + 255) / 256, cap = (size_t)ctx->sm_count * 16;
    return (int)(want < cap ? (want ? want : 1) : cap);
}

bool qparams_ok(int zx, int zw, int zo, int mult, int shift) {
    return zx >= 0 && zx <= 255 && zw >= 0 && zw <= 255 && zo >= 0 && zo <= 255 && mult >= 0 && shift >= 1 && shift <= 62;
}

size_t q_conv_words(int C, int K, int FH, int FW) { return (size_t)blocks_of(K) * blocks_of(C) * FH * FW * 8 * 32; }

}  // namespace

}  // namespace small

using namespace small;

SMALL_API size_t small_q_packed_bytes(int N, int C, int H, int W) { return packed_elems(N, C, H, W); }

SMALL_API int small_q_pack(small_ctx *ctx, const uint8_t *nchw, uint8_t *blk, int N, int C, int H, int W, void *stream) {
    if (!ctx) return SMALL_ERR_NOT_INIT;
    if (!nchw || !blk) return SMALL_ERR_INVALID_ARG;
    if (!aligned16(blk)) return SMALL_ERR_ALIGN;
    if (N < 1 || C < 1 || H < 1 || W < 1 || (long long)H * W > (1ll << 24)) return SMALL_ERR_SHAPE;
    const size_t words = packed_elems(N, C, H, W) / 4;
    if (ranges_overlap(nchw, (size_t)N * C * H * W, blk, words * 4)) return SMALL_ERR_OVERLAP;
    q_pack_kernel<<<grid_for(ctx, words), 256, 0, static_cast<cudaStream_t>(stream)>>>(nchw, reinterpret_cast<uint32_t *>(blk), C, H * W, blocks_of(C), words);
    return check_launch(ctx);
}

SMALL_API int small_q_unpack(small_ctx *ctx, const uint8_t *blk, uint8_t *nchw, int N, int C, int H, int W, void *stream) {
    if (!ctx) return SMALL_ERR_NOT_INIT;
    if (!nchw || !blk) return SMALL_ERR_INVALID_ARG;
    if (!aligned16(blk)) return SMALL_ERR_ALIGN;
    if (N < 1 || C < 1 || H < 1 || W < 1 || (long long)H * W > (1ll << 24)) return SMALL_ERR_SHAPE;
    const size_t words = packed_elems(N, C, H, W) / 4;
    if (ranges_overlap(nchw, (size_t)N * C * H * W, blk, words * 4)) return SMALL_ERR_OVERLAP;
    q_unpack_kernel<<<grid_for(ctx, words), 256, 0, static_cast<cudaStream_t>(stream)>>>(reinterpret_cast<const uint32_t *>(blk), nchw, C, H * W, blocks_of(C), words);
    return check_launch(ctx);
}

SMALL_API size_t small_q_conv_weight_bytes(int C, int K, int FH, int FW) {
    if (C < 1 || K < 1 || FH < 1 || FW < 1) return 0;
    return q_conv_words(C, K, FH, FW) * 4 + ((size_t)K * FH * FW + K) * sizeof(int);      // (the last K words are spare)
}

SMALL_API int small_q_pack_conv_weights(small_ctx *ctx, const uint8_t *w, void *wb, int C, int K, int FH, int FW, void *stream) {
    if (!ctx) return SMALL_ERR_NOT_INIT;
    if (!w || !wb) return SMALL_ERR_INVALID_ARG;
    if (!aligned16(wb)) return SMALL_ERR_ALIGN;
    if (C < 1 || K < 1 || FH < 1 || FW < 1 || (long long)K * FH * FW > (1ll << 28)) return SMALL_ERR_SHAPE;
    if (ranges_overlap(w, (size_t)K * C * FH * FW, wb, small_q_conv_weight_bytes(C, K, FH, FW))) return SMALL_ERR_OVERLAP;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const size_t words = q_conv_words(C, K, FH, FW);
    const int T = FH * FW;
    pack_q_conv_w_kernel<<<grid_for(ctx, words), 256, 0, st>>>(w, static_cast<uint32_t *>(wb), C, K, T, words);
    q_conv_tables_kernel<<<(K * T + 127) / 128, 128, 0, st>>>(w, reinterpret_cast<int *>(static_cast<uint32_t *>(wb) + words), C, K, T);
    return check_launch(ctx);
}

SMALL_API int small_q_conv2d(small_ctx *ctx, const uint8_t *in, const void *w_blk, const int32_t *bias, uint8_t *out,
                             int N, int C, int K, int H, int W, int FH, int FW, int stride, int pt, int pb, int pl, int pr,
                             int z_in, int z_w, int z_out, int mult, int shift, unsigned flags, void *stream) {
    if (!ctx) return SMALL_ERR_NOT_INIT;
    CallOfItsOwn call(ctx);
    if (flags & ~SMALL_RELU) return SMALL_ERR_INVALID_ARG;
    if (!in || !w_blk || !out || !qparams_ok(z_in, z_w, z_out, mult, shift)) return SMALL_ERR_INVALID_ARG;
    if (!aligned16(in) || !aligned16(w_blk) || !aligned16(out) || (bias && (reinterpret_cast<uintptr_t>(bias) & 3u))) return SMALL_ERR_ALIGN;
    Geom g;
    if (int s = make_geom(g, N, C, K, H, W, FH, FW, stride, pt, pb, pl, pr)) return s;
    if ((long long)C * FH * FW > 33000) return SMALL_ERR_SHAPE;      // the raw sums of byte products must stay inside 32 bits
    if (ranges_overlap(in, packed_elems(N, C, H, W), out, packed_elems(N, K, g.OH, g.OW))) return SMALL_ERR_OVERLAP;
    const uint8_t *w = static_cast<const uint8_t *>(w_blk);
    const int *sums = reinterpret_cast<const int *>(w + q_conv_words(C, K, FH, FW) * 4);
    return launch_q_conv(ctx, in, w, sums, bias, out, g, flags & SMALL_RELU, z_in, z_w, z_out, mult, shift, static_cast<cudaStream_t>(stream));
}

SMALL_API size_t small_q_dw_weight_bytes(int C, int FH, int FW) {
    if (C < 1 || FH < 1 || FW < 1) return 0;
    return (size_t)blocks_of(C) * FH * FW * 32;
}

SMALL_API int small_q_pack_dw_weights(small_ctx *ctx, const uint8_t *w, uint8_t *wb, int C, int FH, int FW, void *stream) {
    if (!ctx) return SMALL_ERR_NOT_INIT;
    if (!w || !wb) return SMALL_ERR_INVALID_ARG;
    if (!aligned16(wb)) return SMALL_ERR_ALIGN;
    if (C < 1 || FH < 1 || FW < 1 || (long long)blocks_of(C) * FH * FW * 32 > (1ll << 30)) return SMALL_ERR_SHAPE;
    const int total = (int)small_q_dw_weight_bytes(C, FH, FW);
    if (ranges_overlap(w, (size_t)C * FH * FW, wb, total)) return SMALL_ERR_OVERLAP;
    pack_q_dw_w_kernel<<<(total + 255) / 256, 256, 0, static_cast<cudaStream_t>(stream)>>>(w, wb, C, FH * FW, total);
    return check_launch(ctx);
}

SMALL_API int small_q_dwconv2d(small_ctx *ctx, const uint8_t *in, const uint8_t *w_blk, const int32_t *bias, uint8_t *out,
                               int N, int C, int H, int W, int FH, int FW, int stride, int pt, int pb, int pl, int pr,
                               int z_in, int z_w, int z_out, int mult, int shift, unsigned flags, void *stream) {
    if (!ctx) return SMALL_ERR_NOT_INIT;
    CallOfItsOwn call(ctx);
    if (flags & ~SMALL_RELU) return SMALL_ERR_INVALID_ARG;
    if (!in || !w_blk || !out || !qparams_ok(z_in, z_w, z_out, mult, shift)) return SMALL_ERR_INVALID_ARG;
    if (!aligned16(in) || !aligned16(w_blk) || !aligned16(out) || (bias && (reinterpret_cast<uintptr_t>(bias) & 3u))) return SMALL_ERR_ALIGN;
    Geom g;
    if (int s = make_geom(g, N, C, C, H, W, FH, FW, stride, pt, pb, pl, pr)) return s;
    if ((long long)FH * FW > 33000) return SMALL_ERR_SHAPE;
    if (ranges_overlap(in, packed_elems(N, C, H, W), out, packed_elems(N, C, g.OH, g.OW))) return SMALL_ERR_OVERLAP;
    QPlaneArgs a{reinterpret_cast<const uint32_t *>(in), reinterpret_cast<uint32_t *>(out), reinterpret_cast<const uint32_t *>(w_blk), bias,
                 N, C, g.CB, H, W, FH, FW, stride, pt, pl, g.OH, g.OW, z_in, z_w, z_out, mult, shift, (flags & SMALL_RELU) ? z_out : 0};
    const long long columns = (long long)N * g.CB * g.OW * 8;
    if (FH == 3 && FW == 3 && stride <= 2 && columns * g.OH < (1ll << 31)) {
        // a column is cut into runs of at least four rows as long as that takes the SMs to some 800 threads each
        int segs = (int)(800ll * ctx->sm_count / columns);
        segs = segs < 1 ? 1 : segs > ceil_div(g.OH, 4) ? ceil_div(g.OH, 4) : segs;
        const int R = ceil_div(g.OH, segs);
        segs = ceil_div(g.OH, R);
        const unsigned items = (unsigned)(columns * segs);
        const bool fast = shift >= 32 && shift <= 43;
        launch_kernel(ctx, stride == 1 ? (fast ? q_dw3x3_kernel<1, true> : q_dw3x3_kernel<1, false>) : (fast ? q_dw3x3_kernel<2, true> : q_dw3x3_kernel<2, false>), dim3((items + 127) / 128), dim3(128), 0, static_cast<cudaStream_t>(stream), a, R, (unsigned)segs, items);
        return check_launch(ctx);
    }
    q_dwconv_kernel<<<grid_for(ctx, packed_elems(N, C, g.OH, g.OW) / 4), 256, 0, static_cast<cudaStream_t>(stream)>>>(a);
    return check_launch(ctx);
}

SMALL_API int small_q_maxpool2d(small_ctx *ctx, const uint8_t *in, uint8_t *out, int N, int C, int H, int W, int FH, int FW,
                                int stride, int pt, int pb, int pl, int pr, int z, void *stream) {
    if (!ctx) return SMALL_ERR_NOT_INIT;
    CallOfItsOwn call(ctx);
    if (!in || !out || z < 0 || z > 255) return SMALL_ERR_INVALID_ARG;
    if (!aligned16(in) || !aligned16(out)) return SMALL_ERR_ALIGN;
    Geom g;
    if (int s = make_geom(g, N, C, C, H, W, FH, FW, stride, pt, pb, pl, pr)) return s;
    if (ranges_overlap(in, packed_elems(N, C, H, W), out, packed_elems(N, C, g.OH, g.OW))) return SMALL_ERR_OVERLAP;
    QPlaneArgs a{reinterpret_cast<const uint32_t *>(in), reinterpret_cast<uint32_t *>(out), nullptr, nullptr,
                 N, C, g.CB, H, W, FH, FW, stride, pt, pl, g.OH, g.OW, z, 0, 0, 0, 1, 0};
    const size_t items = packed_elems(N, C, g.OH, g.OW) / 16;
    if (items < (1ull << 31) - 1024 * 1024)
        launch_kernel(ctx, q_maxpool_kernel<unsigned>, dim3(grid_for(ctx, items)), dim3(256), 0, static_cast<cudaStream_t>(stream), a, (unsigned)items);
    else launch_kernel(ctx, q_maxpool_kernel<size_t>, dim3(grid_for(ctx, items)), dim3(256), 0, static_cast<cudaStream_t>(stream), a, items);
    return check_launch(ctx);
}

SMALL_API int small_q_relu(small_ctx *ctx, const uint8_t *in, uint8_t *out, int N, int C, int H, int W, int z, void *stream) {
    if (!ctx) return SMALL_ERR_NOT_INIT;
    if (!in || !out || z < 0 || z > 255) return SMALL_ERR_INVALID_ARG;
    if (!aligned16(in) || !aligned16(out)) return SMALL_ERR_ALIGN;
    const size_t bytes = packed_elems(N, C, H, W);
    if (bytes == 0) return SMALL_ERR_SHAPE;
    if (in != out && ranges_overlap(in, bytes, out, bytes)) return SMALL_ERR_OVERLAP;
    q_relu_kernel<<<grid_for(ctx, bytes / 4), 256, 0, static_cast<cudaStream_t>(stream)>>>(reinterpret_cast<const uint32_t *>(in), reinterpret_cast<uint32_t *>(out),
                                                                                         C, blocks_of(C), H * W, z, bytes / 4);
    return check_launch(ctx);
}
