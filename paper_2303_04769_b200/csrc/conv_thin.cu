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
//     the few lines that an SM's first-level cache has in flight: a line per pixel); from an NCHW tensor, cp.async;
//   * a tile is whole rows of an image, or of several images; of wide planes, some columns of rows (see plan_tiles);
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
    int nb, TH, bands, kgroups;              // images and output rows per tile; row bands of an image; filter groups
    int gt, cbands;                          // column groups (of PIX outputs) of a tile; column bands of an image
    int rows, pitch, plane;                  // shared tile: rows x pitch pairs per (image, channel); plane = rows * pitch
    uint32_t raw_bytes;                      // of the next tile's copy, in front of the planes
    uint32_t by_pitch, by_rows, by_gt;       // divisors as multipliers (see quotient)
    unsigned tiles;                          // (no more than output pixels, whose tensor fits the memory: below 2^31)
    bool relu, accumulate;
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
    // tile t: its first image, its row band and its first column group
    auto place = [&](unsigned t, int &n0, int &band, int &g0) {
        g0 = 0;
        if (a.cbands > 1) { const unsigned q = t / (unsigned)a.cbands; g0 = (int)(t - q * a.cbands) * a.gt; t = q; }
        const unsigned q = t / (unsigned)a.bands;
        band = (int)(t - q * a.bands); n0 = (int)q * a.nb;
    };
    // A tile's pixels, four floats each: [image][row][column], the columns and rows outside the plane zero.
    auto copy = [&](unsigned t) {
        int n0, band, g0;
        place(t, n0, band, g0);
        const int ih0 = band * a.TH * S - a.pt, iw0 = g0 * PIX * S - a.pl;
        if (!a.nchw) {
            if (threadIdx.x == 0) {
                sm100::mbar_expect_tx(full, (uint32_t)(a.nb * a.rows * a.pitch) * 16u);
                sm100::tma_load_5d(raw, &map, full, 0, iw0, ih0, 0, n0);
            }
            return;
        }
        const int total = min(a.nb, a.N - n0) * a.rows * a.pitch;
        const size_t hw = (size_t)a.H * a.W;
        for (int e = threadIdx.x; e < total; e += kThinThreads) {
            int r = quotient(e, a.by_pitch);
            const int gw = e - r * a.pitch + iw0, img = quotient(r, a.by_rows), gh = ih0 + r - img * a.rows;
            const bool in = (unsigned)gh < (unsigned)a.H && (unsigned)gw < (unsigned)a.W;
            const float *p = in ? a.in + ((size_t)(n0 + img) * C * a.H + gh) * a.W + gw : a.in;
#pragma unroll
            for (int c = 0; c < C; ++c)
                asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(raw + (uint32_t)(e * 16 + c * 4)), "l"(in ? p + c * hw : p), "r"(in ? 4 : 0) : "memory");
        }
    };
    uint32_t parity = 0;
    bool alive = true;
    if (blockIdx.x < a.tiles) copy(blockIdx.x);
    for (unsigned t = blockIdx.x; t < a.tiles; t += gridDim.x) {
        int n0, band, g0;
        place(t, n0, band, g0);
        const int imgs = min(a.nb, a.N - n0), oh0 = band * a.TH;
        const int th = min(a.TH, a.OH - oh0), total = imgs * a.rows * a.pitch;
        if (a.nchw) asm volatile("cp.async.wait_all;" ::: "memory");
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
        const int per_img = th * a.gt, items = imgs * per_img;      // (image, output row, column group; some of the last column band's may lie outside)
        for (int it0 = warp * PIECES; it0 < items; it0 += PIECES * (kThinThreads / 32)) {
            const int it = min(it0 + sub, items - 1);
            int img = 0, rg = it;
            if (imgs > 1) { img = it / per_img; rg = it - img * per_img; }
            const int r = quotient(rg, a.by_gt), cg = rg - r * a.gt;
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
            const int oh = oh0 + r, ow0 = (g0 + cg) * PIX;
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

// What a layer needs besides its tensors, made once per shape (a new buffer of a known shape costs a tensor map): the launch, and the
// tensor maps of the inputs seen.
struct ThinPlan { ThinArgs a; ThinKernel kern; dim3 grid; size_t smem; std::unordered_map<const float *, CUtensorMap> maps; };
typedef std::unordered_map<std::string, ThinPlan> ThinCache;

// Columns that `groups` column groups read.
int tile_pitch(const Geom &g, int groups) {
    const int pix = thin_pix(g);
    return (groups - 1) * pix * g.S + 2 * (((pix - 1) * g.S + g.FW + 1) / 2);
}

// The tile: whole rows of an image, several images where planes are small.  Estimated cycles of an SM: its tiles in rounds of as many
// blocks as it holds; a warp alone issues every third or fourth cycle (a window row's reads, then chains of FMAs), more share the
// scheduler (FMA pairs take two slots).
// Of planes so wide that four rows of outputs need more than kRowTile, some columns of the rows: whole rows bring in two or three rows
// for one computed, leave an SM one block from some 300 columns on, and from 640 on can need more than a block has.  These
// tiles are at most kCutTile, so that the registers decide how many blocks an SM holds, and a tile costs some 100 cycles besides (21
// layers, each with up to 60 tiles: the one taken is within 5 % of the best on average).  us, whole rows / columns cut: 3 channels,
// 3 x 3 stride 2, 32 filters on 224 x 224, batch 8 / 64 10.0 / 9.6, 85.1 / 84.2, on 512 x 512, batch 8 113 / 56; stride 1 on 224 x 224, batch 8
// 30.1 / 24.8; 10 x 4, 64 filters on 500 x 128, batch 16 48.5 / 48.9, on 1000 x 257 255 / 158.
constexpr size_t kRowTile = 44 * 1024, kCutTile = 24 * 1024;
bool plan_tiles(const small_ctx *ctx, const Geom &g, int by_regs, ThinArgs &a) {
    const int pix = thin_pix(g), seg2 = ((pix - 1) * g.S + g.FW + 1) / 2, pieces = 32 / thin_lanes(g.K), groups = ceil_div(g.OW, pix);
    const double per_piece = g.C * g.FH * (seg2 + 2.0 * g.FW * pix) + 8.0 * pix;
    auto rows = [&](int th) { return (th - 1) * g.S + g.FH; };
    auto bytes = [&](int nb, int th, int pitch) { return (size_t)nb * rows(th) * pitch * (16 + 8 * g.C); };
    const bool cut = tile_pitch(g, groups) > 256 || bytes(1, g.OH < 4 ? g.OH : 4, tile_pitch(g, groups)) > kRowTile;
    const size_t most = cut ? kCutTile : kRowTile;
    double best = 0.0;
    for (int cbands = 1; cbands <= (cut ? groups : 1); ++cbands) {
        const int gt = ceil_div(groups, cbands), pitch = tile_pitch(g, gt);
        if (ceil_div(groups, gt) != cbands || pitch > 256) continue;
        for (int bands = 1; bands <= g.OH; ++bands) {
            const int th = ceil_div(g.OH, bands);
            if (ceil_div(g.OH, th) != bands || rows(th) > 256) continue;
            if (th < 4 && bands > 1 && best > 0.0) break;
            for (int nb = 1; nb <= (bands * cbands == 1 ? (g.N < 16 ? g.N : 16) : 1) && bytes(nb, th, pitch) <= most; ++nb) {
                const long long tiles = (long long)ceil_div(g.N, nb) * bands * cbands * a.kgroups, on_sm = (tiles + ctx->sm_count - 1) / ctx->sm_count;
                long long held = (long long)(ctx->max_smem_optin / (bytes(nb, th, pitch) + 1024));
                if (held > by_regs) held = by_regs;
                if (held > on_sm) held = on_sm;
                const double work = ceil_div(nb * th * gt, 4 * pieces) * per_piece + (double)nb * rows(th) * pitch * (g.C + 2) * 0.1 + (cut ? 100.0 : 0.0), alone = work * 3.3 + 600.0;
                const double cost = (double)((on_sm + held - 1) / held) * (held * work > alone ? held * work : alone);
                if (best == 0.0 || cost < best) { best = cost; a.TH = th; a.nb = nb; a.bands = bands; a.gt = gt; a.cbands = cbands; a.pitch = pitch; }
            }
        }
    }
    return best > 0.0;
}

}  // namespace

bool conv_thin_supported(const Geom &g) {
    if (g.C > 4 || g.CB != 1) return false;
    if (!pick_thin(g, thin_pix(g), 32)) return false;
    // rows of up to some 850 (four channels) to 3400 columns (one); wider planes take the other kernels
    int pitch = tile_pitch(g, ceil_div(g.OW, thin_pix(g)));
    if (pitch < g.W + g.pl) pitch = (g.W + g.pl + 1) & ~1;
    return (size_t)g.C * g.FH * pitch * sizeof(float) <= 40 * 1024;
}

void free_thin_cache(small_ctx *ctx) {
    delete static_cast<ThinCache *>(ctx->thin_cache);
    ctx->thin_cache = nullptr;
}

static int make_plan(small_ctx *ctx, const Geom &g, bool nchw_in, ThinPlan &p) {
    ThinArgs &a = p.a;
    a = ThinArgs{};
    a.status = ctx->dev_status; a.nchw = nchw_in;
    a.N = g.N; a.K = g.K; a.KB = g.KB; a.H = g.H; a.W = g.W; a.OH = g.OH; a.OW = g.OW; a.pt = g.pt; a.pl = g.pl;
    a.kgroups = ceil_div(g.KB, 2);
    p.kern = pick_thin(g, thin_pix(g), thin_lanes(g.K));
    if (!p.kern) return SMALL_ERR_UNSUPPORTED;
    int by_regs = 1;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&by_regs, p.kern, kThinThreads, 0) != cudaSuccess || by_regs < 1) by_regs = 1;
    if (!plan_tiles(ctx, g, by_regs, a)) return SMALL_ERR_UNSUPPORTED;
    a.rows = (a.TH - 1) * g.S + g.FH;
    a.plane = a.rows * a.pitch;
    a.raw_bytes = (uint32_t)(a.nb * a.plane * 16);
    auto multiplier = [](int d) { return d <= 1 ? 0u : (uint32_t)((1ull << 32) / (unsigned)d) + 1u; };
    a.by_pitch = multiplier(a.pitch); a.by_rows = multiplier(a.rows);
    a.by_gt = multiplier(a.gt);
    a.tiles = (unsigned)((long long)ceil_div(g.N, a.nb) * a.bands * a.cbands);
    p.smem = (size_t)a.nb * a.plane * (16 + 8 * g.C);      // at most kRowTile: within what every launch may have
    // blocks that run at once: the grid is that many (or fewer), each walking the tile list
    int per_sm = 1;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, p.kern, kThinThreads, p.smem) != cudaSuccess || per_sm < 1) per_sm = 1;
    long long gx = (long long)per_sm * ctx->sm_count / a.kgroups;
    if (gx < 1) gx = 1;
    p.grid = dim3(a.tiles < gx ? a.tiles : (unsigned)gx, (unsigned)a.kgroups);
    return SMALL_OK;
}

int launch_conv_thin(small_ctx *ctx, const float *in, const float *w, const float *bias, float *out, const Geom &g,
                     bool relu, bool accumulate, cudaStream_t st, bool nchw_in) {
    if (!conv_thin_supported(g)) return SMALL_ERR_UNSUPPORTED;
    std::string key;
    {
        const int f[] = {g.N, g.C, g.K, g.H, g.W, g.FH, g.FW, g.S, g.pt, g.pb, g.pl, g.pr, nchw_in ? 1 : 0};
        key.append(reinterpret_cast<const char *>(f), sizeof(f));
    }
    if (!ctx->thin_cache) ctx->thin_cache = new ThinCache();
    ThinCache &cache = *static_cast<ThinCache *>(ctx->thin_cache);
    auto it = cache.find(key);
    if (it == cache.end()) {
        ThinPlan made{};
        if (int s = make_plan(ctx, g, nchw_in, made)) return s;
        if (cache.size() >= 512) cache.clear();
        it = cache.emplace(std::move(key), std::move(made)).first;
    }
    ThinPlan &p = it->second;
    const CUtensorMap *map;
    static const CUtensorMap none{};
    if (nchw_in) {
        map = &none;
    } else {
        auto m = p.maps.find(in);
        if (m == p.maps.end()) {
            cuuint64_t dims[5] = {32, (cuuint64_t)g.W, (cuuint64_t)g.H, 1, (cuuint64_t)g.N};
            cuuint64_t strides[4] = {128, (cuuint64_t)g.W * 128, (cuuint64_t)g.H * g.W * 128, (cuuint64_t)g.H * g.W * 128};
            cuuint32_t box[5] = {4, (cuuint32_t)p.a.pitch, (cuuint32_t)p.a.rows, 1, (cuuint32_t)p.a.nb}, es[5] = {1, 1, 1, 1, 1};
            CUtensorMap made;
            CUresult r = reinterpret_cast<sm100::EncodeTiledFn>(ctx->encode_tiled)(&made, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 5, const_cast<float *>(in), dims, strides, box, es,
                             CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_NONE, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
            if (r != CUDA_SUCCESS) { ctx->last_cuda = (int)r; return SMALL_ERR_CUDA; }
            if (p.maps.size() >= 64) p.maps.clear();
            m = p.maps.emplace(in, made).first;
        }
        map = &m->second;
    }
    ThinArgs a = p.a;
    a.in = in; a.w = w; a.bias = bias; a.out = out; a.relu = relu; a.accumulate = accumulate;
    a.wait_iters = ctx->wait_iters; a.late = ctx->dependent == 2;
    launch_kernel(ctx, p.kern, p.grid, dim3(kThinThreads), p.smem, st, *map, a);
    return check_launch(ctx);
}

}  // namespace small
