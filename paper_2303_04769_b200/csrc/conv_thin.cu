// Full channel reduction for layers with at most four input channels (paper Section 3.2 item 4 with a very small
// F_C: the first layer of a network, whose input is an image or a spectrogram).  Such a layer is not a dense
// contraction: its reduction is F_H x F_W x C = 27 or 40 terms, a 32-channel block of the layout holds one to four
// real channels, and a tensor-core K step would carry seven or more zeros for every real product.  It runs on the
// CUDA cores instead, specialised at compile time by (C, F_H, F_W, stride) the way the paper specialises its kernels
// by layer dimensions (Section 4.2):
//   * a lane holds two output channels, so that every FMA instruction is a packed pair (fma.rn.f32x2) of the two; their filters,
//     C x F_H x F_W pairs, live in registers for the whole kernel.  Filters are dealt out so that lanes stand for real ones: a
//     warp holds 64 filters where there are more than 32; up to 32, 16 or 8 filters take 16, 8 or 4 lanes, and the warp works on
//     2, 4 or 8 pieces of the output at once;
//   * the real channels of the next input tile are copied to shared memory while a tile is computed, and then spread over dense
//     planes [image][channel][row][column] with every value twice: a 16-byte read brings two inputs as the pairs that the FMAs
//     take.  The copy is one TMA box of 16 bytes of each pixel's line, zeros outside the plane (as many loads of threads wait for
//     the few lines that an SM's first-level cache has in flight: a line per pixel); from an NCHW tensor, and for very wide planes, cp.async;
//   * a warp computes PIX adjacent output pixels of a row: per window row it reads the (PIX - 1) S + F_W inputs it needs as
//     shared-memory broadcasts and issues PIX x F_W packed FMAs on them.
// Bias, accumulate (the residual join), ReLU and the zero pad lanes are handled as in the other convolution kernels.
// What bounds it.  10 x 4 stem of 64 filters, batch 1024: the FMA pipe (a third of the time busy) and the issue of what stands around it,
// at the 12 warps that its 160 registers leave an SM.  Stems of few filters: the lines read and written (all 128 bytes of a pixel's,
// whatever part of them is real).  Measured called back to back, us, one filter per FMA and a tile's loads in front of its arithmetic /
// now: 10 x 4, 1 -> 64 on 49 x 10, batch 1024 43.2 / 30.7, batch 1 5.8 / 4.6; 3 x 3, 3 -> 16 on 32 x 32, batch 256 20.5 / 16.4, batch 1
// 7.2 / 4.1; 3 x 3 stride 2, 3 -> 8 on 96 x 96, batch 64 24.6 / 20.4, batch 4 11.3 / 6.3; 3 -> 64 on 56 x 56, batch 64 38.9 / 28.7.
#include <string>
#include <unordered_map>

#include "common.cuh"
#include "sm100.cuh"

namespace small {

namespace {

struct ThinArgs {
    const float *in; const float *w; const float *bias; float *out; int *status;
    int N, K, KB, H, W, OH, OW, pt, pl;
    int nb, TH, bands, groups, kgroups;      // images and output rows per tile; tiles per image; column groups; filter groups
    int rows, pitch, plane;                  // shared tile: rows x pitch pairs per (image, channel); plane = rows * pitch
    uint32_t raw_bytes;                      // of the next tile's copy, in front of the planes
    uint32_t by_pitch, by_rows, by_groups;   // divisors as multipliers (see quotient)
    long long tiles;
    bool relu, accumulate;
    bool tma;                                // planes of at most 256 columns with their pads, blocked
    bool nchw;                               // the input is the NCHW tensor float[N][C][H][W] itself (the network's edge)
    uint32_t wait_iters;                     // limit of the bounded waits (polls)
    int late;                                // wait for the kernel in front before reading constants
};

constexpr int kThinThreads = 128;

__device__ __forceinline__ uint64_t thin_fma2(uint64_t a, uint64_t b, uint64_t c) {      // two FMAs
    uint64_t r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ uint64_t pair_of(float x, float y) { return ((uint64_t)__float_as_uint(y) << 32) | __float_as_uint(x); }
// n / d by a multiplication: m = 2^32 / d + 1, 0 for d = 1; exact for n * d < 2^32
__device__ __forceinline__ int quotient(int n, uint32_t m) { return m ? (int)__umulhi((uint32_t)n, m) : n; }

// LANES: lanes that share a piece of the output (a run of PIX pixels): 32 (64 filters, two lines), 16, 8 or 4.
// Blocks per SM that the registers allow: filters, sums and a window row's inputs, and some 24 for everything else.
constexpr int thin_blocks(int taps, int pix, int seg) {
    const int regs = (2 * taps + 2 * pix + 2 * seg + 24 + 7) / 8 * 8;
    return 65536 / kThinThreads / regs < 1 ? 1 : 65536 / kThinThreads / regs;
}
template <int C, int FH, int FW, int S, int PIX, int LANES>
__global__ void __launch_bounds__(kThinThreads, thin_blocks(C *FH *FW, PIX, (PIX - 1) * S + FW + 1)) conv_thin_kernel(const __grid_constant__ CUtensorMap map, const ThinArgs a) {
    extern __shared__ __align__(128) uint8_t smem[];
    __shared__ __align__(8) unsigned long long full_bar;
    __shared__ int abort_flag;
    uint64_t *tile = reinterpret_cast<uint64_t *>(smem + a.raw_bytes);
    constexpr int SEG = (PIX - 1) * S + FW, SEG2 = (SEG + 1) / 2, PIECES = 32 / LANES;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int fl = lane & (LANES - 1), sub = lane / LANES;
    // the lane's two filters: k0 and its neighbour; the filter group is fixed per block: blockIdx.y (LANES = 32: two lines of 32,
    // the last group's second one may not exist)
    const int kb = LANES == 32 ? (int)blockIdx.y * 2 + (fl >> 4) : 0, k0 = kb * 32 + 2 * (fl & 15);
    const bool line_exists = LANES < 32 || kb < a.KB;
    if (a.late) grid_dep_sync();
    // filters: [kb][0][x][y][ci][ko], a pair per 8-byte load (two 4-byte ones put together are put together again at every use)
    uint64_t wr[C][FH][FW];
#pragma unroll
    for (int x = 0; x < FH; ++x)
#pragma unroll
        for (int y = 0; y < FW; ++y)
#pragma unroll
            for (int c = 0; c < C; ++c) {
                const float *at = a.w + ((((size_t)(line_exists ? kb : 0) * FH + x) * FW + y) * 32 + c) * 32;
                wr[c][x][y] = __ldg(reinterpret_cast<const unsigned long long *>(at) + (fl & 15));
            }
    const float b0 = a.bias && k0 < a.K ? a.bias[k0] : 0.0f, b1 = a.bias && k0 + 1 < a.K ? a.bias[k0 + 1] : 0.0f;
    const uint32_t full = sm100::smem_u32(&full_bar);
    if (threadIdx.x == 0) {
        sm100::mbar_init(full, 1);
        abort_flag = 0;
        sm100::mbar_fence_init();
    }
    __syncthreads();
    grid_dep_sync();       // filters and bias are the layer's own constants; the tensors come next
    grid_dep_trigger();

    const uint32_t raw = sm100::smem_u32(smem);
    // A tile's pixels, four floats each: [image][row][column], the columns and rows outside the plane zero.
    auto copy = [&](long long t) {
        const int band = (int)(t % a.bands), n0 = (int)(t / a.bands) * a.nb, ih0 = band * a.TH * S - a.pt;
        if (a.tma) {
            if (threadIdx.x == 0) {
                sm100::mbar_expect_tx(full, (uint32_t)(a.nb * a.rows * a.pitch) * 16u);
                sm100::tma_load_5d(raw, &map, full, 0, -a.pl, ih0, 0, n0);
            }
            return;
        }
        const int total = min(a.nb, a.N - n0) * a.rows * a.pitch;
        const size_t hw = (size_t)a.H * a.W;
        for (int e = threadIdx.x; e < total; e += kThinThreads) {
            int r = quotient(e, a.by_pitch);
            const int gw = e - r * a.pitch - a.pl, img = quotient(r, a.by_rows), gh = ih0 + r - img * a.rows;
            const bool in = (unsigned)gh < (unsigned)a.H && (unsigned)gw < (unsigned)a.W;
            if (!a.nchw) {
                const float *p = in ? a.in + (((size_t)(n0 + img) * a.H + gh) * a.W + gw) * 32 : a.in;
                asm volatile("cp.async.ca.shared.global [%0], [%1], 16, %2;" ::"r"(raw + (uint32_t)(e * 16)), "l"(p), "r"(in ? 16 : 0) : "memory");
                continue;
            }
            const float *p = in ? a.in + ((size_t)(n0 + img) * C * a.H + gh) * a.W + gw : a.in;
#pragma unroll
            for (int c = 0; c < C; ++c)
                asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(raw + (uint32_t)(e * 16 + c * 4)), "l"(in ? p + c * hw : p), "r"(in ? 4 : 0) : "memory");
        }
    };
    uint32_t parity = 0;
    bool alive = true;
    if (blockIdx.x < a.tiles) copy(blockIdx.x);
    for (long long t = blockIdx.x; t < a.tiles; t += gridDim.x) {
        const int band = (int)(t % a.bands), n0 = (int)(t / a.bands) * a.nb, imgs = min(a.nb, a.N - n0), oh0 = band * a.TH;
        const int th = min(a.TH, a.OH - oh0), total = imgs * a.rows * a.pitch;
        if (!a.tma) asm volatile("cp.async.wait_all;" ::: "memory");
        else alive = sm100::mbar_wait_uniform(full, parity, &abort_flag, a.status, a.wait_iters);
        parity ^= 1u;
        if (!__syncthreads_and(alive)) break;  // the tile is there, and the planes are no longer read
        for (int e = threadIdx.x; e < total; e += kThinThreads) {
            int img = 0;
            if (C > 1 && imgs > 1) img = quotient(quotient(e, a.by_pitch), a.by_rows);
            uint64_t *dst = tile + (size_t)img * (C - 1) * a.plane + e;      // (an image's planes take rows * pitch pairs each)
            const float4 v = reinterpret_cast<const float4 *>(smem)[e];
            dst[0] = pair_of(v.x, v.x);
            if (C > 1) dst[a.plane] = pair_of(v.y, v.y);
            if (C > 2) dst[2 * a.plane] = pair_of(v.z, v.z);
            if (C > 3) dst[3 * a.plane] = pair_of(v.w, v.w);
        }
        __syncthreads();
        if (t + gridDim.x < a.tiles) copy(t + gridDim.x);
        const int per_img = th * a.groups, items = imgs * per_img;      // (image, output row, column group)
        for (int it0 = warp * PIECES; it0 < items; it0 += PIECES * (kThinThreads / 32)) {
            const int it = min(it0 + sub, items - 1);
            int img = 0, rg = it;
            if (imgs > 1) { img = it / per_img; rg = it - img * per_img; }
            const int r = quotient(rg, a.by_groups), cg = rg - r * a.groups;
            const uint32_t piece = raw + a.raw_bytes + (uint32_t)(img * C * a.plane + r * S * a.pitch + cg * PIX * S) * 8u;
            uint64_t acc[PIX];
#pragma unroll
            for (int p = 0; p < PIX; ++p) acc[p] = 0ull;
#pragma unroll
            for (int c = 0; c < C; ++c) {
#pragma unroll
                for (int x = 0; x < FH; ++x) {
                    // (PIX - 1) S + FW inputs of this window row; the start is an even number of pairs by construction
                    const uint32_t rowp = piece + (uint32_t)(c * a.plane + x * a.pitch) * 8u;
                    uint64_t seg[2 * SEG2];
                    // (volatile: the compiler would bring many rows forward, at more registers than there are)
#pragma unroll
                    for (int i = 0; i < SEG2; ++i) asm volatile("ld.shared.v2.u64 {%0, %1}, [%2];" : "=l"(seg[2 * i]), "=l"(seg[2 * i + 1]) : "r"(rowp + i * 16));
#pragma unroll
                    for (int y = 0; y < FW; ++y)
#pragma unroll
                        for (int p = 0; p < PIX; ++p) acc[p] = thin_fma2(seg[p * S + y], wr[c][x][y], acc[p]);
                }
            }
            if (it0 + sub >= items || !line_exists) continue;
            const int oh = oh0 + r, ow0 = cg * PIX;
            float *dst = a.out + ((((size_t)(n0 + img) * a.KB + kb) * a.OH + oh) * a.OW + ow0) * 32;
#pragma unroll
            for (int p = 0; p < PIX; ++p) {
                if (ow0 + p >= a.OW) break;
                float v0 = __uint_as_float((uint32_t)acc[p]) + b0, v1 = __uint_as_float((uint32_t)(acc[p] >> 32)) + b1;
                float *line = dst + p * 32;
                float2 *at = reinterpret_cast<float2 *>(line) + (fl & 15);
                if (a.accumulate) { const float2 o = *at; v0 += o.x; v1 += o.y; }
                if (a.relu) { v0 = v0 > 0.f ? v0 : 0.f; v1 = v1 > 0.f ? v1 : 0.f; }
                *at = make_float2(k0 < a.K ? v0 : 0.0f, k0 + 1 < a.K ? v1 : 0.0f);      // pad lanes of the last filter block stay +0
                if (LANES == 8) at[8] = make_float2(0.f, 0.f);          // the line's other lanes
                if (LANES == 4) {
                    reinterpret_cast<float4 *>(line + 8)[fl] = make_float4(0.f, 0.f, 0.f, 0.f);
                    reinterpret_cast<float2 *>(line + 24)[fl] = make_float2(0.f, 0.f);
                }
            }
        }
    }
    // after a timeout: give a copy that may still be in flight a bounded grace period before the block exits
    if (!alive)
        for (uint32_t k = 0; k < (1u << 14); ++k) __nanosleep(200);
}

typedef void (*ThinKernel)(const CUtensorMap, const ThinArgs);

int thin_lanes(int K) { return K <= 8 ? 4 : K <= 16 ? 8 : K <= 32 ? 16 : 32; }

template <int C, int FH, int FW, int S, int PIX>
ThinKernel pick_lanes(int lanes) {
    switch (lanes) {
        case 4: return conv_thin_kernel<C, FH, FW, S, PIX, 4>;
        case 8: return conv_thin_kernel<C, FH, FW, S, PIX, 8>;
        case 16: return conv_thin_kernel<C, FH, FW, S, PIX, 16>;
        default: return conv_thin_kernel<C, FH, FW, S, PIX, 32>;
    }
}

template <int FH, int FW, int S, int PIX>
ThinKernel pick_c(int C, int lanes) {
    switch (C) {
        case 1: return pick_lanes<1, FH, FW, S, PIX>(lanes);
        case 2: return pick_lanes<2, FH, FW, S, PIX>(lanes);
        case 3: return pick_lanes<3, FH, FW, S, PIX>(lanes);
        case 4: return pick_lanes<4, FH, FW, S, PIX>(lanes);
        default: return nullptr;
    }
}

// The compiled specialisations: 3 x 3 windows at strides 1 and 2 for one to four channels, and the 10 x 4 stride-2
// window of a one-channel spectrogram.  PIX = 5 serves planes five outputs wide (stride 2 keeps its reads aligned).
ThinKernel pick_thin(const Geom &g, int pix, int lanes) {
    if (g.FH == 3 && g.FW == 3 && g.S == 1 && pix == 8) return pick_c<3, 3, 1, 8>(g.C, lanes);
    if (g.FH == 3 && g.FW == 3 && g.S == 2 && pix == 8) return pick_c<3, 3, 2, 8>(g.C, lanes);
    if (g.FH == 10 && g.FW == 4 && g.S == 2 && g.C == 1) return pix == 5 ? pick_lanes<1, 10, 4, 2, 5>(lanes) : pick_lanes<1, 10, 4, 2, 8>(lanes);
    return nullptr;
}

int thin_pix(const Geom &g) {
    // five outputs per warp when that wastes fewer lanes of work than eight (stride 2 only: 8-byte aligned reads)
    if (g.S == 2 && g.FH == 10 && ceil_div(g.OW, 5) * 5 < ceil_div(g.OW, 8) * 8) return 5;
    return 8;
}

struct ThinLaunch { CUtensorMap map; ThinArgs a; ThinKernel kern; dim3 grid; size_t smem; };
typedef std::unordered_map<std::string, ThinLaunch> ThinCache;

int thin_pitch(const Geom &g) {
    const int pix = thin_pix(g), groups = ceil_div(g.OW, pix), seg2 = ((pix - 1) * g.S + g.FW + 1) / 2;
    int pitch = (groups - 1) * pix * g.S + 2 * seg2;          // the last column group's reads stay inside the row
    if (pitch < g.W + g.pl) pitch = g.W + g.pl;
    return (pitch + 1) & ~1;
}

}  // namespace

bool conv_thin_supported(const Geom &g) {
    if (g.C > 4 || g.CB != 1) return false;
    if (!pick_thin(g, thin_pix(g), 32)) return false;
    // at least one output row of one image must fit the shared tile
    return (size_t)g.C * g.FH * thin_pitch(g) * sizeof(float) <= 40 * 1024;
}

void free_thin_cache(small_ctx *ctx) {
    delete static_cast<ThinCache *>(ctx->thin_cache);
    ctx->thin_cache = nullptr;
}

int launch_conv_thin(small_ctx *ctx, const float *in, const float *w, const float *bias, float *out, const Geom &g,
                     bool relu, bool accumulate, cudaStream_t st, bool nchw_in) {
    if (!conv_thin_supported(g)) return SMALL_ERR_UNSUPPORTED;
    // a launch seen before (same shape, flags and tensors): everything is ready
    std::string key;
    {
        const int f[] = {g.N, g.C, g.K, g.H, g.W, g.FH, g.FW, g.S, g.pt, g.pb, g.pl, g.pr, relu ? 1 : 0, accumulate ? 1 : 0, nchw_in ? 1 : 0, (int)ctx->wait_iters};
        const void *ptrs[] = {in, w, bias, out};
        key.append(reinterpret_cast<const char *>(f), sizeof(f));
        key.append(reinterpret_cast<const char *>(ptrs), sizeof(ptrs));
    }
    if (!ctx->thin_cache) ctx->thin_cache = new ThinCache();
    ThinCache &cache = *static_cast<ThinCache *>(ctx->thin_cache);
    {
        auto it = cache.find(key);
        if (it != cache.end()) {
            ThinLaunch &L = it->second;
            L.a.late = ctx->dependent == 2;
            launch_kernel(ctx, L.kern, L.grid, dim3(kThinThreads), L.smem, st, L.map, L.a);
            return check_launch(ctx);
        }
    }
    ThinLaunch made{};
    ThinArgs &a = made.a;
    a.late = ctx->dependent == 2;
    a.in = in; a.w = w; a.bias = bias; a.out = out; a.status = ctx->dev_status; a.wait_iters = ctx->wait_iters;
    a.N = g.N; a.K = g.K; a.KB = g.KB; a.H = g.H; a.W = g.W; a.OH = g.OH; a.OW = g.OW; a.pt = g.pt; a.pl = g.pl;
    a.relu = relu; a.accumulate = accumulate; a.nchw = nchw_in;
    a.tma = !nchw_in && thin_pitch(g) <= 256;
    const int pix = thin_pix(g), seg2 = ((pix - 1) * g.S + g.FW + 1) / 2;
    const int lanes = thin_lanes(g.K);
    a.groups = ceil_div(g.OW, pix);
    a.kgroups = ceil_div(g.KB, 2);
    a.pitch = thin_pitch(g);
    const ThinKernel kern = pick_thin(g, pix, lanes);
    if (!kern) return SMALL_ERR_UNSUPPORTED;
    // The tile: whole rows of an image, several images where planes are small.  Estimated cycles of an SM: its tiles in rounds of as many
    // blocks as it holds; a warp alone issues every third or fourth cycle (a window row's reads, then chains of FMAs), more share the
    // scheduler (FMA pairs take two slots).
    const int pieces = 32 / lanes;
    auto pixels = [&](int nb, int th) { return (size_t)nb * ((th - 1) * g.S + g.FH) * a.pitch; };
    auto bytes = [&](int nb, int th) { return pixels(nb, th) * (16 + 8 * g.C); };
    const size_t budget = (bytes(1, 1) > 44 * 1024 ? 240 : 44) * 1024;      // (an output row of one image fits: conv_thin_supported)
    const double per_piece = g.C * g.FH * (seg2 + 2.0 * g.FW * pix) + 8.0 * pix;
    int by_regs = 1;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&by_regs, kern, kThinThreads, 0) != cudaSuccess || by_regs < 1) by_regs = 1;
    double best = 0.0;
    for (int bands = 1; bands <= g.OH; ++bands) {
        const int th = ceil_div(g.OH, bands);
        if (ceil_div(g.OH, th) != bands || (th < 4 && bands > 1 && best > 0.0)) continue;
        for (int nb = 1; nb <= (bands == 1 ? (g.N < 16 ? g.N : 16) : 1) && bytes(nb, th) <= budget; ++nb) {
            if (a.tma && (th - 1) * g.S + g.FH > 256) continue;
            const long long tiles = (long long)ceil_div(g.N, nb) * bands * a.kgroups, on_sm = (tiles + ctx->sm_count - 1) / ctx->sm_count;
            long long held = (long long)(ctx->max_smem_optin / (bytes(nb, th) + 1024));
            if (held > by_regs) held = by_regs;
            if (held < 1) held = 1;
            if (held > on_sm) held = on_sm;
            const double work = ceil_div(nb * th * a.groups, 4 * pieces) * per_piece + pixels(nb, th) * (g.C + 2) * 0.1, alone = work * 3.3 + 600.0;
            const double cost = (double)((on_sm + held - 1) / held) * (held * work > alone ? held * work : alone);
            if (best == 0.0 || cost < best) { best = cost; a.TH = th; a.nb = nb; a.bands = bands; }
        }
    }
    if (best == 0.0) return SMALL_ERR_UNSUPPORTED;
    a.rows = (a.TH - 1) * g.S + g.FH;
    a.plane = a.rows * a.pitch;
    a.raw_bytes = (uint32_t)(pixels(a.nb, a.TH) * 16);
    auto multiplier = [](int d) { return d <= 1 ? 0u : (uint32_t)((1ull << 32) / (unsigned)d) + 1u; };
    a.by_pitch = multiplier(a.pitch); a.by_rows = multiplier(a.rows); a.by_groups = multiplier(a.groups);
    a.tiles = (long long)ceil_div(g.N, a.nb) * a.bands;
    const size_t smem = bytes(a.nb, a.TH);
    if (smem > 48 * 1024) {
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)ctx->max_smem_optin - 1024);
        if (e != cudaSuccess) { ctx->last_cuda = (int)e; return SMALL_ERR_CUDA; }
    }
    // blocks that run at once: the grid is that many (or fewer), each walking the tile list
    int per_sm = 1;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kThinThreads, smem) != cudaSuccess || per_sm < 1) per_sm = 1;
    long long gx_ll = (long long)per_sm * ctx->sm_count / a.kgroups;
    if (gx_ll < 1) gx_ll = 1;
    made.grid = dim3((unsigned)(a.tiles < gx_ll ? a.tiles : gx_ll), (unsigned)a.kgroups);
    made.kern = kern;
    made.smem = smem;
    if (a.tma) {
        cuuint64_t dims[5] = {32, (cuuint64_t)g.W, (cuuint64_t)g.H, 1, (cuuint64_t)g.N};
        cuuint64_t strides[4] = {128, (cuuint64_t)g.W * 128, (cuuint64_t)g.H * g.W * 128, (cuuint64_t)g.H * g.W * 128};
        cuuint32_t box[5] = {4, (cuuint32_t)a.pitch, (cuuint32_t)a.rows, 1, (cuuint32_t)a.nb}, es[5] = {1, 1, 1, 1, 1};
        CUresult r = reinterpret_cast<sm100::EncodeTiledFn>(ctx->encode_tiled)(&made.map, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 5, const_cast<float *>(in), dims, strides, box, es,
                         CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_NONE, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
        if (r != CUDA_SUCCESS) { ctx->last_cuda = (int)r; return SMALL_ERR_CUDA; }
    }
    if (cache.size() >= 4096) cache.clear();
    const ThinLaunch &L = cache[key] = made;
    launch_kernel(ctx, L.kern, L.grid, dim3(kThinThreads), L.smem, st, L.map, L.a);
    return check_launch(ctx);
}

}  // namespace small
