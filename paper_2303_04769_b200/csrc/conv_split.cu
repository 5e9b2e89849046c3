// Full channel reduction over few output pixels on the warp-level tensor core instruction (paper Section 3.2 item 4; Algorithms 1
// and 2), TF32 and 3xTF32, any window and stride: the reduction of an output tile is split over the warps of a thread block.
//
// Why a third tensor-core kernel.  At a batch of one or a few images a layer has 4 to 64 tiles of 16 pixels.  conv_tc.cu and
// conv_mma.cu give a tile's whole reduction to one block's MMA chain - 64 -> 64 on an 8 x 8 plane was two blocks, each behind 216
// MMAs and the 295 KB of filters one SM brought in - while the other SMs idle.  Here the tile is as small as the instruction
// allows (16 pixels x 8 or 16 filters), so that the layer covers the chip, and its (window position, channel block) pairs are dealt to
// up to 16 warps: every operand is loaded at once, straight from L2 into the MMA's registers, no chain is longer than a few MMAs,
// and one pass through shared memory adds up the warps' partial sums in a fixed order.
//
// Operands without shared memory.  A K step's channels may be any eight as long as pixels and filters agree: lane t of a quad takes
// the quarter t of the channel block, which is one or two 16-byte loads per pixel and per filter; four lanes read one 128-byte line.
// 3xTF32: x = x_hi + x_lo split in registers, filters arrive split; the small products have an accumulator of their own.
//
// Bound by latency: launch, two dependent loads from L2, a handful of MMAs, the sum - 1.9 us per call back to back - and behind that by
// the bytes an SM takes from L2.  us, whole-tile kernels and now, 3xTF32, one image: 16 -> 16 3x3 on 32x32 6.3 / 2.1, 32 -> 64 3x3 stride 2
// on 16x16 10.1 / 2.0, 64 -> 64 on 8x8 11.0 / 2.7, 256 -> 256 on 7x7 34.4 / 5.2, 1x1 512 -> 512 on 7x7 15.5 / 3.2.  Short chains also
// round less: relative error of the 256-channel layer 7.2e-6 before, 3.9e-7 now.
#include "common.cuh"

namespace small {

namespace {

struct SplitArgs {
    const float *in, *w_hi, *w_lo, *bias;
    float *out;
    int K, KB, CB, H, W, OH, OW, FH, FW, S, pt, pl;
    int pixels, chunks;          // output pixels of all images; (channel block, window position) pairs
    int relu, accumulate, late;
    // JOIN: a 1x1 layer of other pixels and filters whose result this one is added to
    const float *in2, *w2_hi, *w2_lo, *bias2;
    int CB2, H2, W2, S2;
};

__device__ __forceinline__ void mma_tf32(float (&c)[4], const uint32_t (&a)[4], const uint32_t b0, const uint32_t b1) {
    asm volatile("mma.sync.aligned.m16n8k8.row.col.f32.tf32.tf32.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
                 : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3]) : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// NF: fragments of 8 filters of a block's tile; CW: channels of a block that exist (16: layers of at most 16 channels); JOIN: a residual
// stage's 1x1 shortcut as further steps of the reduction it is added to - no launch of its own, nothing written and read again
template <int NF, int CW, bool X3, bool JOIN>
__global__ void __launch_bounds__(512) conv_split_kernel(const SplitArgs a) {
    constexpr int V = CW / 16;                    // 16-byte loads of a lane per pixel and per filter
    extern __shared__ float2 part[];              // [warp][fragment][row half][lane]
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, warps = blockDim.x >> 5;
    const int g = lane >> 2, t = lane & 3, taps = a.FH * a.FW;
    const int p0 = blockIdx.x * 16, k0 = blockIdx.y * 8 * NF;
    const size_t w_chunk = (size_t)a.KB * 32 * 32;
    const size_t w_lane = (size_t)(k0 + g) * 32 + t * (CW / 4);
    const size_t plane = (size_t)a.H * a.W * 32;

    const int chunks = a.chunks + (JOIN ? a.CB2 : 0);
    int iy[2], ix[2];
    const float *img[2], *img2[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int p = p0 + g + 8 * h, q = p < a.pixels ? p : 0;
        const int n = q / (a.OH * a.OW), r = q - n * a.OH * a.OW, oy = r / a.OW;
        iy[h] = p < a.pixels ? oy * a.S - a.pt : -0x10000000;      // rows of pixels that do not exist are outside the plane
        ix[h] = (r - oy * a.OW) * a.S - a.pl;
        img[h] = a.in + (size_t)n * a.CB * plane + t * (CW / 4);
        img2[h] = JOIN ? a.in2 + ((size_t)n * a.CB2 * a.H2 * a.W2 + (oy * a.W2 + (r - oy * a.OW)) * a.S2) * 32 + t * (CW / 4) : nullptr;
    }
    uint4 wh[NF][V], wl[X3 ? NF : 1][V], px[2][V];
    auto load_w = [&](const int c) {
        const float *h = a.w_hi + (size_t)c * w_chunk + w_lane, *l = X3 ? a.w_lo + (size_t)c * w_chunk + w_lane : h;
        if (JOIN && c >= a.chunks) {
            h = a.w2_hi + (size_t)(c - a.chunks) * w_chunk + w_lane;
            l = X3 ? a.w2_lo + (size_t)(c - a.chunks) * w_chunk + w_lane : h;
        }
#pragma unroll
        for (int n = 0; n < NF; ++n)
#pragma unroll
            for (int v = 0; v < V; ++v) {
                wh[n][v] = *reinterpret_cast<const uint4 *>(h + n * 256 + v * 4);
                if (X3) wl[X3 ? n : 0][v] = *reinterpret_cast<const uint4 *>(l + n * 256 + v * 4);
            }
    };
    auto load_px = [&](const int c) {
        if (JOIN && c >= a.chunks) {              // (pixels that do not exist read those of the first one)
#pragma unroll
            for (int h = 0; h < 2; ++h)
#pragma unroll
                for (int v = 0; v < V; ++v)
                    px[h][v] = *reinterpret_cast<const uint4 *>(img2[h] + (size_t)(c - a.chunks) * a.H2 * a.W2 * 32 + v * 4);
            return;
        }
        const int cb = c / taps, tap = c - cb * taps, dy = tap / a.FW, dx = tap - dy * a.FW;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int y = iy[h] + dy, x = ix[h] + dx;
            const bool in = (unsigned)y < (unsigned)a.H && (unsigned)x < (unsigned)a.W;
            const float *s = img[h] + (size_t)cb * plane + (size_t)(in ? y * a.W + x : 0) * 32;
#pragma unroll
            for (int v = 0; v < V; ++v) px[h][v] = in ? *reinterpret_cast<const uint4 *>(s + v * 4) : make_uint4(0, 0, 0, 0);
        }
    };

    if (a.late) grid_dep_sync();
    if (warp < chunks) load_w(warp);            // the filters are the layer's own constants
    grid_dep_sync();
    grid_dep_trigger();
    if (warp < chunks) load_px(warp);

    float acc[NF][4], small[X3 ? NF : 1][4];
#pragma unroll
    for (int n = 0; n < NF; ++n)
#pragma unroll
        for (int e = 0; e < 4; ++e) { acc[n][e] = 0.0f; if (X3) small[X3 ? n : 0][e] = 0.0f; }
    for (int c = warp; c < chunks; c += warps) {
        uint32_t ah[2 * V][4], al[X3 ? 2 * V : 1][4], bh[2 * V][NF][2], bl[X3 ? 2 * V : 1][X3 ? NF : 1][2];
        // K step s: elements 2 s and 2 s + 1 of a lane's channels
#pragma unroll
        for (int s = 0; s < 2 * V; ++s) {
            const bool z = s & 1;
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const uint4 r = px[h][s >> 1];
                const uint32_t e0 = z ? r.z : r.x, e1 = z ? r.w : r.y;
                // TF32: the MMA reads the leading 11 bits of the raw word.  3xTF32: those bits and the exact residual.
                ah[s][h] = X3 ? e0 & 0xffffe000u : e0;
                ah[s][h + 2] = X3 ? e1 & 0xffffe000u : e1;
                if (X3) {
                    al[X3 ? s : 0][h] = __float_as_uint(__uint_as_float(e0) - __uint_as_float(ah[s][h]));
                    al[X3 ? s : 0][h + 2] = __float_as_uint(__uint_as_float(e1) - __uint_as_float(ah[s][h + 2]));
                }
            }
#pragma unroll
            for (int n = 0; n < NF; ++n) {
                const uint4 r = wh[n][s >> 1];
                bh[s][n][0] = z ? r.z : r.x; bh[s][n][1] = z ? r.w : r.y;
                if (X3) {
                    const uint4 q = wl[X3 ? n : 0][s >> 1];
                    bl[X3 ? s : 0][X3 ? n : 0][0] = z ? q.z : q.x; bl[X3 ? s : 0][X3 ? n : 0][1] = z ? q.w : q.y;
                }
            }
        }
        const int next = c + warps;
        if (next < chunks) { load_w(next); load_px(next); }
#pragma unroll
        for (int s = 0; s < 2 * V; ++s)
#pragma unroll
            for (int n = 0; n < NF; ++n) {
                mma_tf32(acc[n], ah[s], bh[s][n][0], bh[s][n][1]);
                if (X3) {
                    mma_tf32(small[X3 ? n : 0], al[X3 ? s : 0], bh[s][n][0], bh[s][n][1]);
                    mma_tf32(small[X3 ? n : 0], ah[s], bl[X3 ? s : 0][X3 ? n : 0][0], bl[X3 ? s : 0][X3 ? n : 0][1]);
                }
            }
    }
#pragma unroll
    for (int n = 0; n < NF; ++n)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            float2 r = make_float2(acc[n][2 * h], acc[n][2 * h + 1]);
            if (X3) { r.x += small[X3 ? n : 0][2 * h]; r.y += small[X3 ? n : 0][2 * h + 1]; }
            part[((warp * NF + n) * 2 + h) * 32 + lane] = r;
        }
    __syncthreads();

    // accumulator rows lane >> 2 and + 8 are pixels, columns 2 (lane & 3) and + 1 of each fragment filters
    for (int i = threadIdx.x; i < NF * 64; i += blockDim.x) {
        const int p = p0 + ((i >> 5) & 1) * 8 + ((i & 31) >> 2), k = k0 + (i >> 6) * 8 + 2 * (i & 3);
        if (p >= a.pixels) continue;
        const int n = p / (a.OH * a.OW), r = p - n * a.OH * a.OW;
        float *dst = a.out + (((size_t)n * a.KB + (k >> 5)) * a.OH * a.OW + r) * 32 + (k & 31);
        float2 v = a.accumulate ? *reinterpret_cast<const float2 *>(dst) : make_float2(0.0f, 0.0f);
        const float b0 = a.bias && k < a.K ? a.bias[k] : 0.0f, b1 = a.bias && k + 1 < a.K ? a.bias[k + 1] : 0.0f;
        if (JOIN && a.bias2) { if (k < a.K) v.x += a.bias2[k]; if (k + 1 < a.K) v.y += a.bias2[k + 1]; }
        float2 s = part[i];
#pragma unroll 4
        for (int w = 1; w < warps; ++w) { const float2 q = part[w * NF * 64 + i]; s.x += q.x; s.y += q.y; }
        v.x += s.x + b0; v.y += s.y + b1;
        if (a.relu) { v.x = fmaxf(v.x, 0.0f); v.y = fmaxf(v.y, 0.0f); }
        if (k >= a.K) v.x = 0.0f;                 // pad lanes stay +0
        if (k + 1 >= a.K) v.y = 0.0f;
        *reinterpret_cast<float2 *>(dst) = v;
        if (i < 64 && blockIdx.y == gridDim.y - 1)      // filters behind the last tile: pad lanes of the last block
            for (int z = k + 8 * NF; z < a.KB * 32; z += 8) *reinterpret_cast<float2 *>(dst + (z - k)) = make_float2(0.0f, 0.0f);
    }
}

template <int NF, int CW>
void launch_form(small_ctx *ctx, const SplitArgs &a, bool x3, dim3 grid, int warps, cudaStream_t st) {
    const size_t smem = (size_t)warps * NF * 64 * sizeof(float2);
    const auto k = a.in2 ? (x3 ? conv_split_kernel<NF, CW, true, true> : conv_split_kernel<NF, CW, false, true>)
                         : (x3 ? conv_split_kernel<NF, CW, true, false> : conv_split_kernel<NF, CW, false, false>);
    launch_kernel(ctx, k, grid, dim3(32 * warps), smem, st, a);
}

// How a layer is cut: filters of a tile, warps that share its reduction, and the time expected of it in us.
struct SplitPlan { int nf, warps; unsigned px_tiles, k_tiles; double us; };

SplitPlan cut(long long pixels, int K, int chunks, bool narrow, bool x3, int sms) {
    SplitPlan best{};
    for (int nf = 1; nf <= 2; ++nf) {
        if (nf == 2 && K <= 8) break;
        const long long px = (pixels + 15) / 16, kt = (K + 8 * nf - 1) / (8 * nf);
        const int resident = x3 ? (nf == 1 ? 20 : 16) : (nf == 1 ? 26 : 22);      // warps an SM's registers hold
        const double kb = (narrow ? 1.0 : 2.0) * (1.0 + 0.5 * nf * (x3 ? 2 : 1));
        int last = 0;
        for (int rounds = (chunks + 15) / 16; rounds <= chunks; ++rounds) {
            const int warps = (chunks + rounds - 1) / rounds;
            if (warps == last) continue;
            last = warps;
            const int per_sm = resident / warps;       // blocks
            const long long waves = (px * kt + (long long)sms * per_sm - 1) / ((long long)sms * per_sm);
            const long long on_sm = (px * kt + sms - 1) / sms;
            const int busy = (int)(on_sm < per_sm ? on_sm : per_sm) * warps;
            const double t = busy * kb / 80.0;
            // a round is a load from L2 that nothing hides (0.45 us), or the bytes of all resident warps at some 80 a ns
            const double us = 1.3 + (double)waves * (0.3 + rounds * (t > 0.45 ? t : 0.45));
            if (!best.nf || us < best.us) best = SplitPlan{nf, warps, (unsigned)px, (unsigned)kt, us};
        }
    }
    return best;
}

// more: steps besides the layer's own.  Every launch asks: the latest answers are kept by what they depend on.
SplitPlan plan_split(const Geom &g, bool x3, int sms, int more = 0) {
    struct Kept { long long pixels; int K, chunks, narrow, x3, sms; SplitPlan p; };
    static thread_local Kept kept[64];
    const long long pixels = (long long)g.N * g.OH * g.OW;
    const int chunks = g.CB * g.FH * g.FW + more, narrow = g.C <= 16;
    Kept &k = kept[(size_t)(pixels * 31 + g.K * 7 + chunks * 3 + narrow + 2 * x3) % 64];
    if (k.pixels != pixels || k.K != g.K || k.chunks != chunks || k.narrow != narrow || k.x3 != x3 || k.sms != sms)
        k = Kept{pixels, g.K, chunks, narrow, x3, sms, cut(pixels, g.K, chunks, narrow, x3, sms)};
    return k.p;
}

}  // namespace

// Few pixels: where the split cut beats the whole-tile kernels clearly.  Their time hardly depends on the pixels there - one block's
// chain of `chunks` steps (conv_tc.cu 5.7 + 0.18 us a step in TF32, 4.4 + 0.38 in 3xTF32 for 3 x 3; conv_mma.cu 3.4 to 6.2) - while
// this kernel's grows with them.  us, whole-tile against split, batch by batch: 64 -> 64 3x3 on 16x16 in 3xTF32, 1 / 4 / 8 / 16 images
// 11.0 / 11.1 / 11.1 / 11.3 against 2.7 / 4.8 / 8.4 / 13.0, in TF32 9.4 / 9.4 / 9.4 / 9.6 against 2.5 / 4.1 / 7.1 / 10.2; 16 -> 16 on
// 32x32 3xTF32, 1 / 8: 6.3 / 6.4 against 2.1 / 4.7; 256 -> 256 1x1 on 14x14, 1 / 8 / 16: 16.4 / 16.6 / 16.7 against 3.3 / 12.6 / 17.7.
// The estimates are up to 1.7 times off near the line, hence the margin.  What the rule sends here, measured back to back against the
// whole-tile kernel forced on the same call: in 3xTF32 94 layers and batches, none slower by more than 1 %, half of them 2.1 times and
// more faster; in TF32 92, half 1.8 times and more, but three slower, as whole tiles take less there than the estimate says when calls
// overlap: 64 -> 64 3x3 on 16x16, batch 8 7.2 / 8.0, on 8x8, batch 37 7.3 / 8.1, 128 -> 128 on 14x14, batch 4 10.4 / 10.7.
bool conv_split_preferred(const Geom &g, bool x3, bool warp_level, int sms) {
    if ((long long)g.N * g.OH * g.OW > 1 << 20 || (long long)g.H * g.W > 1 << 24 || g.K > 1 << 16) return false;
    const int taps = g.FH * g.FW, chunks = g.CB * taps;
    double whole;
    if (warp_level) whole = taps == 1 ? (x3 ? 3.5 : 3.3) : x3 ? 6.2 : g.C <= 16 ? 4.2 : 5.8;
    else if (taps == 1) whole = x3 ? (5.2 + 0.9 * chunks < 12.5 ? 5.2 + 0.9 * chunks : 12.5) : (5.0 + 0.55 * chunks < 10.0 ? 5.0 + 0.55 * chunks : 10.0);
    else whole = x3 ? 4.4 + 0.38 * chunks : 5.7 + 0.175 * chunks;
    return plan_split(g, x3, sms).us < 0.6 * whole;
}

int launch_conv_split(small_ctx *ctx, const float *in, const float *w_hi, const float *w_lo, const float *bias, float *out,
                      const Geom &g, bool relu, bool accumulate, unsigned mode, cudaStream_t st, const Shortcut *sc) {
    const bool x3 = mode == SMALL_MATH_3XTF32;
    SplitArgs a{in, w_hi, w_lo, bias, out, g.K, g.KB, g.CB, g.H, g.W, g.OH, g.OW, g.FH, g.FW, g.S, g.pt, g.pl,
                g.N * g.OH * g.OW, g.CB * g.FH * g.FW, relu, accumulate, ctx->dependent == 2, nullptr, nullptr, nullptr, nullptr, 0, 0, 0, 0};
    if (sc) {
        a.in2 = sc->in; a.w2_hi = sc->w_hi; a.w2_lo = sc->w_lo; a.bias2 = sc->bias;
        a.CB2 = sc->g.CB; a.H2 = sc->g.H; a.W2 = sc->g.W; a.S2 = sc->g.S;
    }
    const SplitPlan p = plan_split(g, x3, ctx->sm_count, a.CB2);
    const dim3 grid(p.px_tiles, p.k_tiles);
    if (g.C <= 16 && (!sc || sc->g.C <= 16)) { if (p.nf == 2) launch_form<2, 16>(ctx, a, x3, grid, p.warps, st); else launch_form<1, 16>(ctx, a, x3, grid, p.warps, st); }
    else if (p.nf == 2) launch_form<2, 32>(ctx, a, x3, grid, p.warps, st);
    else launch_form<1, 32>(ctx, a, x3, grid, p.warps, st);
    return check_launch(ctx);
}

}  // namespace small
