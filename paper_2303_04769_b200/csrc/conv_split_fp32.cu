// Full channel reduction in FP32 over few output pixels (paper Algorithms 1 and 2), any window and stride: the reduction of an output
// tile is split over the warps of a thread block.
//
// Why a third FP32 kernel.  conv_direct.cu and conv_fp32.cu give a tile of 64 and more pixels x 32 filters its whole reduction in one
// block, channel block after channel block with barriers between: at a batch of a few images that chain is the layer's time (64 -> 64
// 3x3 on 8x8: 27 us whether 1 or 37 images) while most of the chip idles.  Here a tile is 8 pixels x 32 filters and its (channel
// block, window position) pairs are dealt to up to 16 warps; one pass through shared memory adds up the warps' partial sums in a fixed
// order.
//
// Within a warp a lane computes 4 filters x all pixels of the tile over a quarter of the channels.  What a lane is handed from cache
// and shared memory is the limit - 32 lanes x 4 bytes a clock for an SM, broadcast or not, against 128 FMAs - so a value has to serve
// several FMAs: with a filter per lane, every pixel handed to all of them, the kernel took three times as long.  The pixels go through
// the warp's own piece of shared memory, channel by channel, so that 16 bytes are two packed pairs of pixels: an FMA instruction does
// two (fma.rn.f32x2, rounded as two FMAs).  The next step's pixels and filters are on their way while a step is computed, filters into
// the registers of those just used.
//
// us, whole-tile kernels and now, one image: 16 -> 16 3x3 on 32x32 10.3 / 2.5, 64 -> 64 on 8x8 27.1 / 3.7, 256 -> 256 on 7x7 104 / 9.1,
// 64 -> 128 1x1 stride 2 on 56x56 18.6 / 2.8, 512 -> 512 1x1 on 7x7 41 / 3.6.  Small partial sums also round less: relative error of the
// 256-channel 3x3 layer 8.2e-7 before, 1.4e-7 now.
#include "common.cuh"

namespace small {

namespace {

struct SplitFp32Args {
    const float *in, *w, *bias;
    float *out;
    int K, KB, CB, H, W, OH, OW, FH, FW, S, pt, pl;
    int pixels, chunks;          // output pixels of all images; (channel block, window position) pairs
    int relu, accumulate, late;
    // DW: a depthwise 3x3 in front of a 1x1 layer; H, W, S, pt, pl above are its input's and its own, FH = FW = 1
    const float *dw, *dw_bias;
    int C, dw_relu;
    // JOIN: a 1x1 layer of other pixels and filters whose result this one is added to
    const float *in2, *w2, *bias2;
    int CB2, H2, W2, S2;
};

__device__ __forceinline__ void fma2(uint64_t &c, uint64_t a, uint64_t b) { asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(c) : "l"(a), "l"(b)); }
__device__ __forceinline__ float2 plus(uint64_t a, uint64_t b) {
    float2 x, y;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(x.x), "=f"(x.y) : "l"(a));
    asm("mov.b64 {%0, %1}, %2;" : "=f"(y.x), "=f"(y.y) : "l"(b));
    return make_float2(x.x + y.x, x.y + y.y);
}

constexpr int P = 8;             // pixels of a tile: 16 take twice as long per step and leave room for fewer warps
constexpr int kMaxWarps = 16;

// CI: channels of a block that are computed (16: layers of at most 16 channels).  DW: the pixels are a depthwise 3x3's results, which a
// lane computes where it would load them - once more for every block of 32 filters, in place of a launch and a tensor.  JOIN: a residual
// stage's 1x1 shortcut as further steps of the reduction it is added to.
template <int CI>
struct Room { static constexpr int kFloats = CI * (P + 4) > P * 32 ? CI * (P + 4) : P * 32; };     // of a warp

template <int CI, bool DW, bool JOIN>
__global__ void __launch_bounds__(32 * kMaxWarps) conv_split_fp32_kernel(const SplitFp32Args a) {
    constexpr int PITCH = P + 4, NX = P * CI / 128, NC = CI / 4;    // floats from channel to channel; 16-byte pixel loads of a lane; its channels
    extern __shared__ __align__(16) float smem[];                   // a warp's pixels [channel][pixel], then its sums [pixel][filter]
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, warps = blockDim.x >> 5, taps = a.FH * a.FW;
    const int p0 = blockIdx.x * P, kb = blockIdx.y, quarter = lane >> 3;
    float *mine = smem + warp * Room<CI>::kFloats;
    const size_t plane = (size_t)a.H * a.W * 32;
    const float *w_lane = a.w + (size_t)kb * a.chunks * 1024 + quarter * NC * 32 + (lane & 7) * 4;

    // the pixel this lane brings, 16 bytes of four channels at a time
    const int p = p0 + lane % P, q = p < a.pixels ? p : 0;
    const int n = q / (a.OH * a.OW), r = q - n * a.OH * a.OW, oy = r / a.OW;
    const int iy = p < a.pixels ? oy * a.S - a.pt : -0x10000000;       // rows of pixels that do not exist are outside the plane
    const int ix = (r - oy * a.OW) * a.S - a.pl;
    const float *img = a.in + (size_t)n * a.CB * plane;

    const int chunks = a.chunks + (JOIN ? a.CB2 : 0);
    const float *w2_lane = JOIN ? a.w2 + (size_t)kb * a.CB2 * 1024 + quarter * NC * 32 + (lane & 7) * 4 : nullptr;
    const float *img2 = JOIN ? a.in2 + ((size_t)n * a.CB2 * a.H2 * a.W2 + (oy * a.W2 + (r - oy * a.OW)) * a.S2) * 32 + lane / P * 4 : nullptr;

    float4 px[NX], w[NC];
    auto load_w = [&](const int c, const int i) {
        const float *f = JOIN && c >= a.chunks ? w2_lane + (size_t)(c - a.chunks) * 1024 : w_lane + (size_t)c * 1024;
        w[i] = *reinterpret_cast<const float4 *>(f + i * 32);
    };
    auto load_px = [&](const int c) {
        if constexpr (DW) {
            const float *s = img + (size_t)c * plane + lane / P * 4, *f = a.dw + (size_t)c * 288 + lane / P * 4;
#pragma unroll
            for (int j = 0; j < NX; ++j) {
                const int ch = c * 32 + (lane / P + j * (32 / P)) * 4;
                float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
                for (int tap = 0; tap < 9; ++tap) {
                    const int y = iy + tap / 3, x = ix + tap % 3;
                    const bool in = (unsigned)y < (unsigned)a.H && (unsigned)x < (unsigned)a.W;
                    const float4 d = in ? *reinterpret_cast<const float4 *>(s + (size_t)(y * a.W + x) * 32 + j * (32 / P) * 4) : make_float4(0.f, 0.f, 0.f, 0.f);
                    const float4 g = *reinterpret_cast<const float4 *>(f + tap * 32 + j * (32 / P) * 4);
                    v.x = fmaf(d.x, g.x, v.x); v.y = fmaf(d.y, g.y, v.y); v.z = fmaf(d.z, g.z, v.z); v.w = fmaf(d.w, g.w, v.w);
                }
                if (a.dw_bias) {                  // C entries
                    if (ch < a.C) v.x += a.dw_bias[ch];
                    if (ch + 1 < a.C) v.y += a.dw_bias[ch + 1];
                    if (ch + 2 < a.C) v.z += a.dw_bias[ch + 2];
                    if (ch + 3 < a.C) v.w += a.dw_bias[ch + 3];
                }
                if (a.dw_relu) { v.x = v.x > 0.f ? v.x : 0.f; v.y = v.y > 0.f ? v.y : 0.f; v.z = v.z > 0.f ? v.z : 0.f; v.w = v.w > 0.f ? v.w : 0.f; }
                px[j] = v;
            }
            return;
        }
        if (JOIN && c >= a.chunks) {              // (a pixel that does not exist reads the first one's)
#pragma unroll
            for (int j = 0; j < NX; ++j)
                px[j] = *reinterpret_cast<const float4 *>(img2 + (size_t)(c - a.chunks) * a.H2 * a.W2 * 32 + j * (32 / P) * 4);
            return;
        }
        const int cb = c / taps, tap = c - cb * taps, dy = tap / a.FW, y = iy + dy, x = ix + tap - dy * a.FW;
        const bool in = (unsigned)y < (unsigned)a.H && (unsigned)x < (unsigned)a.W;
        const float *s = img + (size_t)cb * plane + (size_t)(in ? y * a.W + x : 0) * 32 + lane / P * 4;
#pragma unroll
        for (int j = 0; j < NX; ++j) px[j] = in ? *reinterpret_cast<const float4 *>(s + j * (32 / P) * 4) : make_float4(0.f, 0.f, 0.f, 0.f);
    };

    if (a.late) grid_dep_sync();
    if (warp < chunks)                          // the filters are the layer's own constants
#pragma unroll
        for (int i = 0; i < NC; ++i) load_w(warp, i);
    grid_dep_sync();
    grid_dep_trigger();
    if (warp < chunks) load_px(warp);

    uint64_t acc[P / 2][4];                       // pairs of pixels x filters
#pragma unroll
    for (int j = 0; j < P / 2; ++j)
#pragma unroll
        for (int f = 0; f < 4; ++f) acc[j][f] = 0;
    for (int c = warp; c < chunks; c += warps) {
        const int next = c + warps;
        float *x_store = mine + lane / P * 4 * PITCH + lane % P;
#pragma unroll
        for (int j = 0; j < NX; ++j) {
            float *d = x_store + j * (32 / P) * 4 * PITCH;
            d[0] = px[j].x; d[PITCH] = px[j].y; d[2 * PITCH] = px[j].z; d[3 * PITCH] = px[j].w;
        }
        __syncwarp();
        if (next < chunks) load_px(next);
        const float *x_lane = mine + quarter * NC * PITCH;
#pragma unroll
        for (int i = 0; i < NC; ++i) {
            uint64_t ww[4];
            asm("mov.b64 %0, {%1, %1};" : "=l"(ww[0]) : "f"(w[i].x));
            asm("mov.b64 %0, {%1, %1};" : "=l"(ww[1]) : "f"(w[i].y));
            asm("mov.b64 %0, {%1, %1};" : "=l"(ww[2]) : "f"(w[i].z));
            asm("mov.b64 %0, {%1, %1};" : "=l"(ww[3]) : "f"(w[i].w));
#pragma unroll
            for (int j = 0; j < P / 4; ++j) {
                const ulonglong2 x = *reinterpret_cast<const ulonglong2 *>(x_lane + i * PITCH + 4 * j);
#pragma unroll
                for (int f = 0; f < 4; ++f) { fma2(acc[2 * j][f], x.x, ww[f]); fma2(acc[2 * j + 1][f], x.y, ww[f]); }
            }
            if (next < chunks) load_w(next, i);
        }
        __syncwarp();
    }
    // the quarters' sums: each hands three quarters of its pixels over and keeps the totals of one
    float2 half[P / 4][4], sum[P / 8][4];
#pragma unroll
    for (int j = 0; j < P / 4; ++j)
#pragma unroll
        for (int f = 0; f < 4; ++f) {
            const bool up = lane & 16;
            half[j][f] = plus(up ? acc[j + P / 4][f] : acc[j][f], __shfl_xor_sync(0xffffffffu, up ? acc[j][f] : acc[j + P / 4][f], 16));
        }
#pragma unroll
    for (int j = 0; j < P / 8; ++j)
#pragma unroll
        for (int f = 0; f < 4; ++f) {
            const bool up = lane & 8;
            const float2 give = up ? half[j][f] : half[j + P / 8][f], keep = up ? half[j + P / 8][f] : half[j][f];
            sum[j][f].x = keep.x + __shfl_xor_sync(0xffffffffu, give.x, 8);
            sum[j][f].y = keep.y + __shfl_xor_sync(0xffffffffu, give.y, 8);
        }
    const int from = ((lane & 16) ? P / 2 : 0) + ((lane & 8) ? P / 4 : 0);
#pragma unroll
    for (int j = 0; j < P / 8; ++j) {
        float *d = mine + (from + 2 * j) * 32 + (lane & 7) * 4;
        *reinterpret_cast<float4 *>(d) = make_float4(sum[j][0].x, sum[j][1].x, sum[j][2].x, sum[j][3].x);
        *reinterpret_cast<float4 *>(d + 32) = make_float4(sum[j][0].y, sum[j][1].y, sum[j][2].y, sum[j][3].y);
    }
    __syncthreads();

    const int k = kb * 32 + lane;
    const float bv = (a.bias && k < a.K ? a.bias[k] : 0.0f) + (JOIN && a.bias2 && k < a.K ? a.bias2[k] : 0.0f);
    for (int i = warp; i < P && p0 + i < a.pixels; i += warps) {
        const int m = (p0 + i) / (a.OH * a.OW);
        float *dst = a.out + (((size_t)m * a.KB + kb) * a.OH * a.OW + (p0 + i - m * a.OH * a.OW)) * 32 + lane;
        float s = smem[i * 32 + lane];
#pragma unroll 4
        for (int u = 1; u < warps; ++u) s += smem[u * Room<CI>::kFloats + i * 32 + lane];
        s += bv;
        if (a.accumulate) s += *dst;
        if (a.relu) s = s > 0.f ? s : 0.f;
        *dst = k < a.K ? s : 0.0f;                // pad lanes stay +0
    }
}

template <bool DW, bool JOIN>
void launch_form(small_ctx *ctx, const SplitFp32Args &a, bool narrow, dim3 grid, int warps, cudaStream_t st) {
    if (narrow) launch_kernel(ctx, conv_split_fp32_kernel<16, DW, JOIN>, grid, dim3(32 * warps), (size_t)warps * Room<16>::kFloats * sizeof(float), st, a);
    else launch_kernel(ctx, conv_split_fp32_kernel<32, DW, JOIN>, grid, dim3(32 * warps), (size_t)warps * Room<32>::kFloats * sizeof(float), st, a);
}

// How a layer is cut: warps that share a tile's reduction, and the time expected of it in us.
struct SplitFp32Plan { int warps; unsigned px_tiles; double us; };

SplitFp32Plan cut(long long pixels, int KB, int chunks, bool narrow, bool dw, int sms) {
    SplitFp32Plan best{};
    const int resident = narrow ? 20 : 16;         // warps an SM's registers hold
    const long long px = (pixels + P - 1) / P, tiles = px * KB, on_sm = (tiles + sms - 1) / sms;
    // a round: its latency, and what a resident warp is handed from cache and shared memory (a depthwise layer's pixels and filters
    // are another 36 loads of 16 bytes per lane)
    const double latency = dw ? 1.2 : narrow ? 0.42 : 0.46, warp = (narrow ? 0.04 : 0.062) * (dw ? 6.0 : 1.0);
    int last = 0;
    for (int rounds = (chunks + kMaxWarps - 1) / kMaxWarps; rounds <= chunks; ++rounds) {
        const int warps = (chunks + rounds - 1) / rounds;
        if (warps == last) continue;
        last = warps;
        const int per_sm = resident / warps;       // blocks
        const long long waves = (tiles + (long long)sms * per_sm - 1) / ((long long)sms * per_sm);
        const int busy = (int)(on_sm < per_sm ? on_sm : per_sm) * warps;
        const double us = 0.6 + (double)waves * (1.2 + rounds * (latency + warp * busy));
        if (!best.warps || us < best.us) best = SplitFp32Plan{warps, (unsigned)px, us};
    }
    return best;
}

// more: steps besides the layer's own.  Every launch asks: the latest answers are kept by what they depend on.
SplitFp32Plan plan_split_fp32(const Geom &g, int sms, bool dw, int more = 0) {
    struct Kept { long long pixels; int KB, chunks, narrow, dw, sms; SplitFp32Plan p; };
    static thread_local Kept kept[64];
    const long long pixels = (long long)g.N * g.OH * g.OW;
    const int chunks = g.CB * g.FH * g.FW + more, narrow = g.C <= 16;
    Kept &k = kept[(size_t)(pixels * 31 + g.KB * 7 + chunks * 3 + narrow + 2 * dw) % 64];
    if (k.pixels != pixels || k.KB != g.KB || k.chunks != chunks || k.narrow != narrow || k.dw != dw || k.sms != sms)
        k = Kept{pixels, g.KB, chunks, narrow, dw, sms, cut(pixels, g.KB, chunks, narrow, dw, sms)};
    return k.p;
}

bool fits(const Geom &g) { return (long long)g.N * g.OH * g.OW <= 1 << 20 && (long long)g.H * g.W <= 1 << 24 && g.K <= 1 << 16; }

}  // namespace

// Few pixels: where the split cut beats the whole-tile kernels clearly.  Those take a tile's whole reduction one channel after the
// other, 4.5 + 0.043 us per channel and window position for windows of several positions and some 5 + 0.07 for 1 x 1, at any number of
// pixels that fits the chip at once.  us, whole-tile against split, 1 / 4 / 16 / 37 images: 64 -> 64 3x3 on 16x16 30.8 / 30.9 / 31.1 / 31.3
// against 3.8 / 5.6 / 16.0 / 30.2; 16 -> 16 on 32x32 10.3 / 10.5 / 10.6 against 2.5 / 5.6 / 17.8; 256 -> 256 1x1 on 14x14 32.8 / 32.9 / 30.8 /
// 39.2 against 3.5 / 9.0 / 29.3 / 64.2; 64 -> 64 1x1 on 28x28 9.8 / 10.0 / 11.1 / 15.1 against 2.4 / 4.0 / 10.1 / 20.5.  Of 108
// layers and batches that the rule sends here none is slower than with the whole-tile kernel forced, the least is 1.4 times faster.
double conv_split_fp32_us(const Geom &g, int sms) {
    if (!fits(g)) return 0.0;
    const int taps = g.FH * g.FW;
    const double whole = taps > 1 ? 4.5 + 0.043 * g.C * taps : 5.0 + 0.07 * g.C < 40.0 ? 5.0 + 0.07 * g.C : 40.0;
    const double us = plan_split_fp32(g, sms, false).us;
    return us < 0.75 * whole ? us : 0.0;
}

int launch_conv_split_fp32(small_ctx *ctx, const float *in, const float *w, const float *bias, float *out, const Geom &g,
                           bool relu, bool accumulate, cudaStream_t st, const Shortcut *sc) {
    SplitFp32Args a{in, w, bias, out, g.K, g.KB, g.CB, g.H, g.W, g.OH, g.OW, g.FH, g.FW, g.S, g.pt, g.pl,
                    g.N * g.OH * g.OW, g.CB * g.FH * g.FW, relu, accumulate, ctx->dependent == 2, nullptr, nullptr, g.C, 0, nullptr, nullptr, nullptr, 0, 0, 0, 0};
    if (sc) { a.in2 = sc->in; a.w2 = sc->w; a.bias2 = sc->bias; a.CB2 = sc->g.CB; a.H2 = sc->g.H; a.W2 = sc->g.W; a.S2 = sc->g.S; }
    const SplitFp32Plan p = plan_split_fp32(g, ctx->sm_count, false, a.CB2);
    const dim3 grid(p.px_tiles, (unsigned)g.KB);
    if (sc) launch_form<false, true>(ctx, a, g.C <= 16 && sc->g.C <= 16, grid, p.warps, st);
    else launch_form<false, false>(ctx, a, g.C <= 16, grid, p.warps, st);
    return check_launch(ctx);
}

// One launch instead of two costs the host half, and the device a depthwise layer per 32 filters.  us per pair of the keyword-spotting
// network (64 channels on 25x5), two launches against one, 1 / 8 / 16 / 37 images: 4.2 / 4.8 / 5.8 / 6.9 against 3.5 / 4.4 / 6.1 / 8.4; a
// depthwise layer on its own takes some 2.8, and 0.8 more are given for the host's time.
double split_pair_us(const Geom &gp, int sms) {
    if (!fits(gp)) return 0.0;
    const double us = plan_split_fp32(gp, sms, true).us;
    return us < 3.6 + plan_split_fp32(gp, sms, false).us ? us : 0.0;
}

int launch_split_pair(small_ctx *ctx, const float *in, const float *dw, const float *dw_bias, bool dw_relu, const float *w, const float *bias,
                      float *out, const Geom &gd, const Geom &gp, bool relu, cudaStream_t st) {
    const SplitFp32Args a{in, w, bias, out, gp.K, gp.KB, gp.CB, gd.H, gd.W, gp.OH, gp.OW, 1, 1, gd.S, gd.pt, gd.pl,
                          gp.N * gp.OH * gp.OW, gp.CB, relu, 0, ctx->dependent == 2, dw, dw_bias, gp.C, dw_relu, nullptr, nullptr, nullptr, 0, 0, 0, 0};
    const SplitFp32Plan p = plan_split_fp32(gp, ctx->sm_count, true);
    launch_form<true, false>(ctx, a, gp.C <= 16, dim3(p.px_tiles, (unsigned)gp.KB), p.warps, st);
    return check_launch(ctx);
}

}  // namespace small
