// A run of depthwise 3x3 -> 1x1 pairs as ONE kernel (paper Section 6, the abstract fused layer, over whole stacks of a
// depthwise-separable network), the 1x1 layers on the tensor cores (tcgen05), with the global average pool and the classifier
// behind them where the run ends in those.  A thread block keeps one image in shared memory from the run's input to its end:
//
//   plane        [channel block][pixel][36 floats]: 32 channels and four floats apart, so that eight neighbouring pixels' 16-byte
//                pieces lie in eight bank groups.  TMA brings a run's input there (a box of 36 floats over rows of 32: what lies
//                outside the tensor is filled with zeros); behind every pair the epilogue writes the pair's result there.
//   depthwise    eight warps; a thread holds R x NC outputs of four channels, walks down the input rows under them and adds each
//                value to every output it belongs to, in packed pairs of FMAs.  All results of a layer stay in registers until
//                every warp has read the plane; then they replace it, as the MMAs' operand (128-byte swizzle): per channel block
//                the TF32 part of each pixel and, behind the last pixel, the residuals (3xTF32).
//   1x1 layer    One warp streams the filters through a ring of stages by TMA, one (128 filters, channel block) box at a time, across
//                the layers' and images' ends; another issues the MMAs.  Either the filters are the MMA's M rows and the pixels its
//                N (few pixels: an MMA costs (128 + N) / 4 cycles), in 3xTF32 w_hi against [x_hi; x_lo] and w_lo against x_hi; or
//                the pixels are M and the filters N ([w_hi; w_lo] against x_hi, w_hi against x_lo), where a layer has at
//                most 64 filters and 65 to 128 pixels.
//   epilogue     the eight warps again: tensor memory -> registers, + bias, ReLU -> plane; behind the last pair global memory, or
//                the sums over the pixels and the full reduction on them.
//
// Why.  Launched one by one the layers of such a network take 6 to 10 us each whatever the batch below some 64 images, most of it
// start-up, first loads and the drain; at larger batches each pair moves its tensors out of the SMs and back twice.  Here a pair
// costs its depthwise, MMAs and epilogue in sequence, 2.5 to 3.5 us, and two blocks on an SM fill each other's gaps.  Measured called
// directly, us, before and now: keyword-spotting network 3xTF32 batch 1 41 / 21, 148 47 / 27, 1024 177 / 127 (TF32 161 / 116),
// depthwise-separable network (its last ten pairs) batch 1 124 / 76, 64 178 / 120 (TF32 157 / 114).
// What bounds it (64 channels on 25 x 5, 3xTF32, cycles of a block alone on its SM): depthwise 1700 and 1000 to store the operand, issue
// slots of two warps per scheduler and the latencies between them; 16 MMAs 1450, 900 of them the tensor pipe's; epilogue 1350.  With two
// blocks on an SM (batch 1024) no unit is full: of some 5800 cycles per image and pair shared memory answers the warps in 1870, issue
// slots are 42 % used, the FMA pipe 21 %, the tensor pipe 15 %; barriers between a pair's steps are the largest stall.  Measured and not kept: 16 warps a block (fewer
// registers: spills, 141 us at batch 1024), a warp of their own for copies or MMAs (a ninth warp leaves 96 registers at two blocks on
// an SM), layers' parameters in shared memory, the next layer's depthwise filters loaded during the MMAs.
#include <cuda.h>

#include <cstring>
#include <memory>
#include <type_traits>
#include <unordered_map>
#include <vector>

#include "common.cuh"
#include "sm100.cuh"

namespace small {

namespace {

using namespace sm100;

constexpr int kThreads = 256, kMma = 4, kCopy = 5;           // two of the eight warps issue MMAs and copies besides their share
constexpr int kMaxPairs = 14, kMaxRing = 8;
constexpr uint32_t kSpin = 1u << 15;                         // polls without back-off on the layer-to-layer critical path
constexpr int kMaxBlocks = 8;                                // channel blocks of a layer
// Runs of at least three pairs.  (Two gain as well; they stay with the layer kernels and the on-chip kernel, whose lines were measured on them.)
constexpr int kMinPairs = 3;

struct PairOp {
    int C, K, CB, KB, H, W, OH, OW, pt, pl;
    int px, pxp;                    // output pixels; rounded up to 16
    int tile, ncg, units;           // depthwise: compiled tile, groups of columns, threads with work
    int pix_m, wide;                // orientation; 3xTF32 with filters on M: [x_hi; x_lo] as one operand
    int m_tiles, rows;              // filters on M: tiles of 128; filter rows of a box
    int dw_relu, relu, b_at, dwb_at;// biases in shared memory (floats)
    uint32_t in_stride, op_stride, out_stride;      // bytes between channel blocks: plane read, operand, plane written
    uint32_t d_cols;                // tensor-memory columns of a tile of filters
    uint32_t idesc, idesc_wide;
    const float *dw_w, *dw_bias, *bias;
};

struct Maps { CUtensorMap in; CUtensorMap w[kMaxPairs][2]; };

struct Args {
    PairOp p[kMaxPairs];
    int n, N;
    int ring, ring2, grow_at, tmem_cols;
    uint32_t stage_bytes, extra_off;
    uint32_t plane_off, dww_off, dww_bytes, bias_off, head_off, ctrl_off;
    float *out; int *status;
    // classifier behind the run (head_K > 0): packed FP32 filters [KB][CB][32][32]
    const float *head_w, *head_bias; int head_K, head_relu, head_b_at;
    uint32_t wait_iters;
    int late;                       // wait for the kernel in front before reading constants
};

__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {      // two FMAs
    uint64_t r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
// the same in every lane, as the compiler can tell: operands of copies and MMAs then stay in uniform registers
__device__ __forceinline__ uint32_t uniform(uint32_t v) { return __shfl_sync(0xffffffffu, v, 0); }
__device__ __forceinline__ float lo_of(uint64_t v) { return __uint_as_float((uint32_t)v); }
__device__ __forceinline__ float hi_of(uint64_t v) { return __uint_as_float((uint32_t)(v >> 32)); }

// The depthwise tiles that are compiled: columns x rows of outputs a thread holds, the stride; `full`: the columns are the whole
// plane's with pads of one, so that what lies outside is known at compile time.  Compiled for planes of five columns; planes of other
// widths take the tiles of three, and what full tiles of four, six or seven columns would give was not measured.
struct DwTile { int nc, r, s; bool full; };
constexpr DwTile kTiles[] = {{5, 2, 1, true}, {3, 2, 1, false}, {3, 2, 2, false}, {3, 1, 2, false}, {3, 4, 1, false}, {5, 4, 1, true}};
constexpr int kTileCount = sizeof(kTiles) / sizeof(kTiles[0]), kTilesTwo = 4;      // two blocks on an SM: the first four (registers)
constexpr uint32_t kPitch = 144;                             // bytes of a pixel of the plane

__device__ __forceinline__ ulonglong2 lds16(uint32_t addr) {
    ulonglong2 v;
    asm volatile("ld.shared.v2.u64 {%0, %1}, [%2];" : "=l"(v.x), "=l"(v.y) : "r"(addr));
    return v;
}
__device__ __forceinline__ ulonglong2 lds16_if(uint32_t addr, bool ok) {      // zero otherwise
    ulonglong2 v;
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %3, 0;\n\tmov.b64 %0, 0;\n\tmov.b64 %1, 0;\n\t@p ld.shared.v2.u64 {%0, %1}, [%2];\n\t}"
                 : "=l"(v.x), "=l"(v.y) : "r"(addr), "r"((uint32_t)ok));
    return v;
}
__device__ __forceinline__ void sts16(uint32_t addr, float x, float y, float z, float w) {
    asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "f"(x), "f"(y), "f"(z), "f"(w) : "memory");
}
__device__ __forceinline__ float hi_tf32(float x) { return __uint_as_float(__float_as_uint(x) & 0xffffe000u); }

// One layer's depthwise part: this thread's outputs from the plane into registers; when every thread has read, into the operand.
template <bool X3, int TILE>
__device__ __forceinline__ void depthwise(const PairOp &o, const uint32_t plane, const uint32_t wts, const uint32_t bias, const bool alive) {
    constexpr int NC = kTiles[TILE].nc, R = kTiles[TILE].r, S = kTiles[TILE].s;
    constexpr bool FULL = kTiles[TILE].full;
    constexpr int COLS = (NC - 1) * S + 3, ROWS = (R - 1) * S + 3;
    const int quads = o.CB * 8, t = threadIdx.x;
    const int rest = t / quads, qd = t - rest * quads, rs = FULL ? rest : rest / o.ncg, cg = FULL ? 0 : rest - rs * o.ncg;
    const int cb = qd >> 3, j = qd & 7, oh0 = rs * R, ow0 = cg * NC;      // four channels, the first output
    const bool work = alive && t < o.units;
    uint64_t acc[R][NC][2];
    if (work) {
        const uint32_t wt = wts + (uint32_t)(cb * 9 * 128 + j * 16);
        {
            const ulonglong2 b = lds16(bias + (uint32_t)(o.dwb_at + qd * 4) * 4u);
#pragma unroll
            for (int r = 0; r < R; ++r)
#pragma unroll
                for (int c = 0; c < NC; ++c) { acc[r][c][0] = b.x; acc[r][c][1] = b.y; }
        }
        const int W = o.W, H = o.H;
        const int ih0 = oh0 * S - o.pt, iw0 = ow0 * S - (FULL ? 1 : o.pl);
        ulonglong2 w[3][3];                            // the window's rows, each loaded when the first input row needs it
        uint32_t row_at = plane + (uint32_t)cb * o.in_stride + j * 16 + (uint32_t)((ih0 * W + iw0) * (int)kPitch);      // (outside: not read)
#pragma unroll
        for (int i = 0; i < ROWS; ++i) {
            if (i < 3)
#pragma unroll
                for (int y = 0; y < 3; ++y) w[i][y] = lds16(wt + (i * 3 + y) * 128);
            const bool row = (unsigned)(ih0 + i) < (unsigned)H;
            ulonglong2 v[COLS];
#pragma unroll
            for (int c = 0; c < COLS; ++c) {
                if (FULL && (c == 0 || c == COLS - 1)) continue;
                v[c] = lds16_if(row_at + c * kPitch, row && (FULL || (unsigned)(iw0 + c) < (unsigned)W));
            }
            row_at += (uint32_t)W * kPitch;
#pragma unroll
            for (int c = 0; c < COLS; ++c) {
                if (FULL && (c == 0 || c == COLS - 1)) continue;
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    const int x = i - r * S;
                    if (x < 0 || x > 2) continue;
#pragma unroll
                    for (int n = 0; n < NC; ++n) {
                        const int y = c - n * S;
                        if (y < 0 || y > 2) continue;
                        acc[r][n][0] = fma2(v[c].x, w[x][y].x, acc[r][n][0]);
                        acc[r][n][1] = fma2(v[c].y, w[x][y].y, acc[r][n][1]);
                    }
                }
            }
        }
    }
    __syncthreads();                                   // the plane has been read by everyone: the operand takes its place
    if (work) {
        const uint32_t dst = plane + (uint32_t)cb * o.op_stride, res = (uint32_t)o.pxp * 128u;
        const int OW = o.OW, OH = o.OH;
        const bool relu = o.dw_relu;
#pragma unroll
        for (int r = 0; r < R; ++r)
#pragma unroll
            for (int n = 0; n < NC; ++n) {
                if (oh0 + r >= OH || (!FULL && ow0 + n >= OW)) continue;
                const int p = (oh0 + r) * OW + ow0 + n;
                float f[4] = {lo_of(acc[r][n][0]), hi_of(acc[r][n][0]), lo_of(acc[r][n][1]), hi_of(acc[r][n][1])};
                if (relu) {
#pragma unroll
                    for (int e = 0; e < 4; ++e) f[e] = fmaxf(f[e], 0.f);
                }
                const uint32_t at = dst + (uint32_t)p * 128u + ((uint32_t)(j ^ (p & 7)) << 4);
                if (X3) {
                    sts16(at, hi_tf32(f[0]), hi_tf32(f[1]), hi_tf32(f[2]), hi_tf32(f[3]));
                    sts16(at + res, f[0] - hi_tf32(f[0]), f[1] - hi_tf32(f[1]), f[2] - hi_tf32(f[2]), f[3] - hi_tf32(f[3]));
                } else {
                    sts16(at, f[0], f[1], f[2], f[3]);
                }
            }
    }
}

// 32 columns of a thread's tensor-memory lane (TWO: of two groups of columns, added up).
template <bool TWO>
__device__ __forceinline__ void read_columns(const uint32_t t0, const uint32_t t1, float (&v)[32]) {
    if (!TWO) return tmem_ld32(t0, v);
    float u[32];
    tmem_ld32x2(t0, t1, v, u);
#pragma unroll
    for (int e = 0; e < 32; ++e) v[e] += u[e];
}

// A pair's result: accumulators -> + bias, ReLU -> plane (or global memory behind the last pair: `out` is the image's tensor).
// `sums`: the sums over the pixels instead, per filter, in four parts of 256.  The warps of a quarter of the tensor-memory lanes
// share out the columns.  ReLU is a maximum with 0, and without one the maximum is with NaN, which leaves numbers and NaNs as they are
// (that with -infinity makes numbers of NaNs).  Pad filters are products of zeros, a NaN where a channel is infinite: with 0, they stay +0.
template <bool X3>
__device__ __forceinline__ void epilogue(const PairOp &o, const uint32_t tmem, const uint32_t plane, float *out, float *sums, const float *bias_s) {
    constexpr int G = 2, CW = 32;                         // warps of a quarter; columns read at a time
    const int lane = threadIdx.x & 31, warp = warp_index(), quarter = warp & 3, group = warp >> 2;
    const uint32_t lanes = (uint32_t)(quarter * 32) << 16;
    const float floor = o.relu ? 0.0f : __int_as_float(0x7fffffff);
    const int px = o.px, rows = o.rows, out_stride = (int)o.out_stride, b_at = o.b_at;
    if (o.pix_m) {
        // lane = pixel, CW filters at a time
        const int p = quarter * 32 + lane;
        for (int k = group * CW; k < rows; k += G * CW) {
            const float4 *b4 = reinterpret_cast<const float4 *>(bias_s + b_at + k);
            float v[CW];
            read_columns<X3>(tmem + lanes + (uint32_t)k, tmem + lanes + (uint32_t)(rows + k), v);
#pragma unroll
            for (int i = 0; i < CW / 4; ++i) {
                const float4 b = b4[i];
                v[4 * i] = fmaxf(v[4 * i] + b.x, floor); v[4 * i + 1] = fmaxf(v[4 * i + 1] + b.y, floor);
                v[4 * i + 2] = fmaxf(v[4 * i + 2] + b.z, floor); v[4 * i + 3] = fmaxf(v[4 * i + 3] + b.w, floor);
            }
            if (k + CW > o.K)
#pragma unroll
                for (int e = 0; e < CW; ++e) v[e] = k + e < o.K ? v[e] : 0.0f;
            if (sums) {
                // over the warp's pixels: halves change places until a lane holds one filter's sum
#pragma unroll
                for (int e = 0; e < CW; ++e) v[e] = p < px ? v[e] : 0.0f;
#pragma unroll
                for (int w = CW / 2; w > 0; w >>= 1)
#pragma unroll
                    for (int e = 0; e < w; ++e) {
                        const float mine = lane & w ? v[e + w] : v[e], other = lane & w ? v[e] : v[e + w];
                        v[e] = mine + __shfl_xor_sync(0xffffffffu, other, w);
                    }
                sums[quarter * 256 + k + (lane & (CW - 1))] = v[0];
            } else if (p < px) {
                const int jj = k >> 5, c = k & 31;
                const uint32_t row = plane + (uint32_t)(jj * out_stride + p * (int)kPitch + c * 4);
                float4 *line = reinterpret_cast<float4 *>(out + ((size_t)jj * px + p) * 32 + c);
#pragma unroll
                for (int i = 0; i < CW / 4; ++i) {
                    if (out) line[i] = make_float4(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]);
                    else sts16(row + i * 16, v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]);
                }
            }
        }
        return;
    }
    const int part = (px + 8 * G - 1) / (8 * G) * 8, p_from = group * part, p_to = p_from + part < px ? p_from + part : px;      // this warp's pixels
    for (int mt = 0; mt < o.m_tiles; ++mt) {
        const int kb = mt * 4 + quarter;
        if (kb >= o.KB) continue;
        const uint32_t d = tmem + lanes + (uint32_t)mt * o.d_cols;
        const float b = bias_s[b_at + kb * 32 + lane];
        const float least = kb * 32 + lane < o.K ? floor : 0.0f;
        const uint32_t blk = plane + (uint32_t)(kb * out_stride + lane * 4);
        float *line = out + (size_t)kb * px * 32 + lane;
        float s[4] = {0.f, 0.f, 0.f, 0.f};
        // (columns past the pixels are read and not used: the plan allocates 32 more)
        for (int p0 = p_from; p0 < p_to; p0 += CW) {
            float v[CW];
            if (X3 && o.wide) read_columns<true>(d + (uint32_t)p0, d + (uint32_t)(o.pxp + p0), v);
            else read_columns<false>(d + (uint32_t)p0, 0, v);
#pragma unroll
            for (int e = 0; e < CW; ++e) v[e] = fmaxf(v[e] + b, least);
            const int left = p_to - p0;
            if (sums) {
#pragma unroll
                for (int e = 0; e < CW; ++e) s[e & 3] += e < left ? v[e] : 0.0f;
            } else if (out) {
#pragma unroll
                for (int e = 0; e < CW; ++e) st_global_if(line + (size_t)(p0 + e) * 32, v[e], e < left);
            } else {
                const uint32_t at = blk + (uint32_t)p0 * kPitch;
#pragma unroll
                for (int e = 0; e < CW; ++e)
                    asm volatile("{\n\t.reg .pred p;\n\tsetp.lt.s32 p, %2, %3;\n\t@p st.shared.f32 [%0], %1;\n\t}" ::"r"(at + e * kPitch), "f"(v[e]), "r"(e), "r"(left) : "memory");
            }
        }
        if (sums) {
            sums[group * 256 + kb * 32 + lane] = (s[0] + s[1]) + (s[2] + s[3]);
            sums[(group + 2) * 256 + kb * 32 + lane] = 0.0f;
        }
    }
}

template <bool X3, int PER_SM>
__global__ void __launch_bounds__(256, PER_SM) sep_chain_kernel(const __grid_constant__ Maps maps, const __grid_constant__ Args a) {
    extern __shared__ uint8_t smem_raw[];
    const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    uint8_t *base_ptr = smem_raw + (base - smem_u32(smem_raw));
    const uint32_t plane = base + a.plane_off;
    const float *bias_s = reinterpret_cast<const float *>(base_ptr + a.bias_off);
    float *head_s = reinterpret_cast<float *>(base_ptr + a.head_off);       // sums [4][256], partials [8][32]
    const uint32_t ctrl = base + a.ctrl_off;
    const uint32_t bar_ring_full = ctrl, bar_ring_empty = ctrl + 8 * kMaxRing, bar_dww = ctrl + 16 * kMaxRing, bar_img = bar_dww + 16;
    volatile uint32_t *tmem_slot = reinterpret_cast<volatile uint32_t *>(base_ptr + a.ctrl_off + 16 * kMaxRing + 64);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(base_ptr + a.ctrl_off + 16 * kMaxRing + 68);
    const int warp = warp_index(), lane = threadIdx.x & 31;

    if (threadIdx.x == 0) {
        for (int s = 0; s < kMaxRing; ++s) { mbar_init(bar_ring_full + 8 * s, 1); mbar_init(bar_ring_empty + 8 * s, 1); }
        mbar_init(bar_dww, 1); mbar_init(bar_dww + 8, 1); mbar_init(bar_img, 1);
        *abort_flag = 0;
        mbar_fence_init();
    }
    if (a.late) grid_dep_sync();
    {   // biases of every layer and of the head, zero in the pad lanes (the layers' own constants); copies that nothing waits for one by one
        auto bring = [&](int at, const float *src, int real, int n) {
            for (int i = threadIdx.x; i < n; i += kThreads) {
                const bool ok = src && i < real;
                asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(base + a.bias_off + (uint32_t)(at + i) * 4u), "l"(ok ? src + i : reinterpret_cast<const float *>(a.status)), "r"(ok ? 4 : 0) : "memory");
            }
        };
        for (int l = 0; l < a.n; ++l) {
            const PairOp &o = a.p[l];
            bring(o.dwb_at, o.dw_bias, o.C, o.CB * 32);
            bring(o.b_at, o.bias, o.K, o.KB * 32);
        }
        bring(a.head_b_at, a.head_bias, a.head_K, (a.head_K + 31) & ~31);
        asm volatile("cp.async.wait_all;" ::: "memory");
    }
    if (warp == 0) tmem_alloc(smem_u32(const_cast<uint32_t *>(tmem_slot)), (uint32_t)a.tmem_cols);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = uniform(*tmem_slot);
    grid_dep_sync();
    grid_dep_trigger();

    // One warp issues the MMAs and one the copies, each as a uniform warp whose thread is elected at the instruction.  What is copied
    // next goes out as soon as its place is free: a box behind the MMAs of the one it replaces, a layer's depthwise filters two layers
    // ahead, the next image behind an image's last MMAs.
    uint32_t armed = 0, parity = 0;              // copies started and their phases: bits 0-7 ring stages, 8-9 depthwise filters, 10 image
    bool alive = true;
    auto copy_image = [&](int n) {
        const PairOp &o = a.p[0];
        if (elect_one()) {
            mbar_expect_tx(bar_img, (uint32_t)(o.CB * o.H * o.W) * kPitch);
            for (int cb = 0; cb < o.CB; ++cb) tma_load_5d(plane + cb * o.in_stride, &maps.in, bar_img, 0, 0, 0, cb, n);
        }
        __syncwarp();
        parity ^= (armed >> 10 & 1u) << 10;
        armed |= 1u << 10;
    };
    auto copy_dww = [&](int l, uint32_t d) {
        const uint32_t bytes = (uint32_t)a.p[l].CB * 1152u, bar = bar_dww + 8 * d;
        if (elect_one()) {
            mbar_expect_tx(bar, bytes);
            bulk_load(base + a.dww_off + d * a.dww_bytes, a.p[l].dw_w, bytes, bar);
        }
        __syncwarp();
        parity ^= (armed >> (8 + d) & 1u) << (8 + d);
        armed |= 1u << (8 + d);
    };
    // The ring: box i of the block's stream lies at position i mod `ring`.  Where a block has one image and the later layers need less
    // of the plane, the ring grows by the stages that fit there (a.ring2) before layer a.grow_at: behind the boxes in flight.
    int ring = a.ring, rot = 0, cq = 0, pq = 0;           // positions of the box multiplied (or handed back) next and of the one copied next
    uint32_t used = 0;                                    // per stage: parity of that use
    auto stage_at = [&](int q) { return q >= a.ring ? q : q + rot >= a.ring ? q + rot - a.ring : q + rot; };
    auto place_of = [&](int st) { return base + (st < a.ring ? (uint32_t)st * a.stage_bytes : a.extra_off + (uint32_t)(st - a.ring) * a.stage_bytes); };
    int bn = blockIdx.x, bl = 0, bm = 0, bc = 0;          // the box that is copied next
    auto copy_box = [&]() {
        if (bn >= a.N) return;
        const PairOp &o = a.p[bl];
        const int st = stage_at(pq);
        const uint32_t box = (uint32_t)o.rows * 128u, dst = place_of(st), bar = bar_ring_full + 8 * st;
        if (elect_one()) {
            mbar_expect_tx(bar, X3 ? 2 * box : box);
            tma_load_3d(dst, &maps.w[bl][0], bar, 0, bm * 128, bc);
            if (X3) tma_load_3d(dst + box, &maps.w[bl][1], bar, 0, bm * 128, bc);
        }
        __syncwarp();
        parity ^= (armed >> st & 1u) << st;
        armed |= 1u << st;
        if (++pq == ring) pq = 0;
        if (++bc == o.CB) {
            bc = 0;
            if (++bm == o.m_tiles) { bm = 0; if (++bl == a.n) { bl = 0; bn += gridDim.x; } }
        }
    };
    // One layer's MMAs.  FORM 0: pixels on M; 1: filters on M (3xTF32: against [x_hi; x_lo]); 2: filters on M, three MMAs per K step
    auto mmas = [&](auto form, const PairOp &o) {
        constexpr int FORM = decltype(form)::value;
        const uint32_t elected = elect_one();
        const uint32_t x_step = o.op_stride >> 4, x_res = (uint32_t)o.pxp * 8u, w_res = (uint32_t)o.rows * 8u;
        const uint32_t idesc = o.idesc, idesc_wide = o.idesc_wide;
        const int CB = o.CB, boxes = CB * o.m_tiles;
        uint32_t dt = tmem, x = smem_desc_lo(plane), last = 0, last_ph = 0;
        for (int i = 0, cb = 0; i < boxes; ++i) {
            const int st = stage_at(cq);
            const uint32_t w = uniform(smem_desc_lo(place_of(st))), xs = uniform(x), ds = uniform(dt);
            alive = mbar_wait_uniform<kSpin>(bar_ring_full + 8 * st, used >> st & 1u, abort_flag, a.status, a.wait_iters);
            if (!alive) return;
            if (elected) {
#pragma unroll
                for (uint32_t k = 0; k < 8; k += 2) {
                    const uint32_t acc = k == 0 ? (uint32_t)cb : 1u;
                    if (FORM == 0) {
                        mma_tf32(ds, xs + k, w + k, kDescHi, idesc_wide, acc);
                        if (X3) mma_tf32(ds, xs + x_res + k, w + k, kDescHi, idesc, 1u);
                    } else if (FORM == 1) {
                        mma_tf32(ds, w + k, xs + k, kDescHi, idesc_wide, acc);
                        if (X3) mma_tf32(ds, w + w_res + k, xs + k, kDescHi, idesc, 1u);
                    } else {
                        mma_tf32(ds, w + k, xs + x_res + k, kDescHi, idesc, acc);      // small terms first
                        mma_tf32(ds, w + w_res + k, xs + k, kDescHi, idesc, 1u);
                        mma_tf32(ds, w + k, xs + k, kDescHi, idesc, 1u);
                    }
                }
                mma_commit(bar_ring_empty + 8 * st);
            }
            __syncwarp();
            last = bar_ring_empty + 8 * st; last_ph = used >> st & 1u;
            used ^= 1u << st;
            if (++cq == ring) cq = 0;
            x += x_step;
            if (++cb == CB) { cb = 0; x = smem_desc_lo(plane); dt += o.d_cols; }
        }
        alive = mbar_wait_uniform<kSpin>(last, last_ph, abort_flag, a.status, a.wait_iters);      // the last box's MMAs are the layer's
    };
    // Meanwhile: the places of a layer's boxes but the last are filled again.
    auto refill = [&](const PairOp &o) {
        const int boxes = o.CB * o.m_tiles;
        for (int i = 0; i < boxes; ++i) {
            const int st = stage_at(cq);
            if (i < boxes - 1) {
                alive = mbar_wait_uniform<kSpin>(bar_ring_empty + 8 * st, used >> st & 1u, abort_flag, a.status, a.wait_iters);
                if (!alive) return;
                copy_box();
            }
            used ^= 1u << st;
            if (++cq == ring) cq = 0;
        }
    };

    if (warp == kCopy) {
        copy_image(bn);
        copy_dww(0, 0);
        copy_dww(1, 1);
        for (int i = 0; i < a.ring; ++i) copy_box();
    }
    uint32_t iph = 0, d = 0, dph = 0;
    // (the barriers are passed in any case, also after a timeout)
    for (int n = blockIdx.x; n < a.N; n += gridDim.x) {
        for (int l = 0; l < a.n; ++l) {
            const PairOp &o = a.p[l];
            if (warp == kMma && alive) {
                if (l == 0) alive = mbar_wait_uniform<kSpin>(bar_img, iph, abort_flag, a.status, a.wait_iters);
                if (alive) alive = mbar_wait_uniform<kSpin>(bar_dww + 8 * d, dph, abort_flag, a.status, a.wait_iters);
            }
            __syncthreads();                              // also: every value of the plane is in place
            alive = __all_sync(0xffffffffu, *abort_flag == 0);
            const uint32_t wts = base + a.dww_off + d * a.dww_bytes, bias = base + a.bias_off;
            if (o.tile == 0) depthwise<X3, 0>(o, plane, wts, bias, alive);
            else if (o.tile == 1) depthwise<X3, 1>(o, plane, wts, bias, alive);
            else if (o.tile == 2) depthwise<X3, 2>(o, plane, wts, bias, alive);
            else if (PER_SM == 2 || o.tile == 3) depthwise<X3, 3>(o, plane, wts, bias, alive);
            else if (o.tile == 4) depthwise<X3, 4>(o, plane, wts, bias, alive);
            else depthwise<X3, 5>(o, plane, wts, bias, alive);
            const uint32_t d_of_layer = d;
            if ((d ^= 1u) == 0u) dph ^= 1u;
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");      // the operand is read by the tensor core
            tc_fence_before();
            __syncthreads();
            if (warp == kMma && alive) {
                tc_fence_after();
                if (o.pix_m) mmas(std::integral_constant<int, 0>{}, o);
                else if (!X3 || o.wide) mmas(std::integral_constant<int, 1>{}, o);
                else mmas(std::integral_constant<int, 2>{}, o);
            }
            if (warp == kCopy && alive) {
                // the depthwise filters of the layer after next take the place of this one's, which every warp has read
                const bool next = l + 2 >= a.n;
                if (!next || n + (int)gridDim.x < a.N) copy_dww(next ? l + 2 - a.n : l + 2, d_of_layer);
                refill(o);
            }
            __syncthreads();
            alive = __all_sync(0xffffffffu, *abort_flag == 0);
            tc_fence_after();
            if (warp == kCopy && alive && l == a.n - 1 && n + (int)gridDim.x < a.N) copy_image(n + gridDim.x);
            if (alive) {
                const bool last = l == a.n - 1;
                epilogue<X3>(o, tmem, plane, last && !a.head_K ? a.out + (size_t)n * o.KB * o.px * 32 : nullptr, last && a.head_K ? head_s : nullptr, bias_s);
            }
            if (l + 1 == a.grow_at) {                     // (the boxes in flight come first, then the new stages)
                rot = stage_at(cq);
                ring = a.ring2; cq = 0; pq = a.ring - 1;
            }
            if (warp == kCopy && alive)                   // in the place of the layer's last box
                for (int i = l + 1 == a.grow_at ? a.ring : ring; i <= ring; ++i) copy_box();
        }
        iph ^= 1u;
        if (a.head_K) {
            // warps share out the averages' rows of the classifier (the first eight are on their way meanwhile); the first adds up
            const PairOp &o = a.p[a.n - 1];
            const int C = o.KB * 32, KB = (a.head_K + 31) >> 5;
            float *sum = head_s + 1024, w[8];
            const float *wt = a.head_w + warp * 32 + lane;
#pragma unroll
            for (int i = 0; i < 8; ++i) w[i] = warp + 8 * i < C ? __ldg(wt + i * 256) : 0.0f;
            __syncthreads();
            if ((int)threadIdx.x < C) {
                const int c = threadIdx.x;
                head_s[c] = ((head_s[c] + head_s[256 + c]) + (head_s[512 + c] + head_s[768 + c])) / (float)o.px;
            }
            __syncthreads();
            for (int kb = 0; kb < KB; ++kb, wt += C * 32) {
                float v = 0.0f;
                int c = warp;
                if (kb == 0) {
#pragma unroll
                    for (int i = 0; i < 8; ++i) v = fmaf(warp + 8 * i < C ? head_s[warp + 8 * i] : 0.0f, w[i], v);
                    c += 64;
                } else {
                    __syncthreads();
                }
#pragma unroll 8
                for (; c < C; c += 8) v = fmaf(head_s[c], __ldg(wt + (c - warp) * 32), v);
                sum[warp * 32 + lane] = v;
                __syncthreads();
                if (warp == 0) {
                    const int k = kb * 32 + lane;
                    v = bias_s[a.head_b_at + k];
#pragma unroll
                    for (int i = 0; i < 8; ++i) v += sum[i * 32 + lane];
                    if (a.head_relu) v = v > 0.f ? v : 0.f;
                    if (alive) a.out[((size_t)n * KB + kb) * 32 + lane] = k < a.head_K ? v : 0.0f;
                }
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (*abort_flag && warp == kCopy && lane == 0)            // a role gave up: let the copies in flight land before the block exits
        for (int i = 0; i < 11; ++i)
            if (armed >> i & 1u) {
                const uint32_t bar = i < 8 ? bar_ring_full + 8 * i : i < 10 ? bar_dww + 8 * (i - 8) : bar_img;
                for (uint32_t it = 0; it < a.wait_iters && !mbar_try_wait(bar, parity >> i & 1u); ++it) __nanosleep(200);
            }
    __syncthreads();
    if (warp == 0) {
        tc_fence_after();
        tmem_dealloc(tmem, (uint32_t)a.tmem_cols);
    }
}

// ---------------------------------------------------------------------------------------------- host side
struct Plan {
    Args a;
    int pairs, layers;               // pairs taken; layers of the list they and the head cover
    size_t smem;
    int per_sm;
    unsigned math;
};

uint32_t round_up(uint32_t v, uint32_t to) { return (v + to - 1) / to * to; }

// The pair of layers at `A`, whose input plane is `o` of the run; false where it does not fit.
bool plan_pair(const small_layer &A, const small_layer &Bn, int N, bool x3, int tile_count, PairOp &o) {
    Geom g;
    if (make_geom(g, N, A.C, A.C, A.H, A.W, 3, 3, A.stride, A.pad_t, A.pad_b, A.pad_l, A.pad_r)) return false;
    o = PairOp{};
    o.C = A.C; o.K = Bn.K; o.CB = g.CB; o.KB = blocks_of(Bn.K); o.H = g.H; o.W = g.W; o.OH = g.OH; o.OW = g.OW; o.pt = g.pt; o.pl = g.pl;
    if (o.CB > kMaxBlocks || o.KB > kMaxBlocks || o.H > 256 || o.W > 256 || (long long)o.H * o.W > 2048 || (long long)o.OH * o.OW > 256) return false;
    o.px = o.OH * o.OW; o.pxp = (int)round_up((uint32_t)o.px, 16);
    // depthwise tile: one per thread; the one that keeps a thread's work smallest
    int best = 0;
    o.tile = -1;
    for (int i = 0; i < tile_count; ++i) {
        const DwTile &t = kTiles[i];
        if (t.s != A.stride || (t.full && (g.W != t.nc || g.OW != t.nc || g.pl != 1))) continue;
        const int ncg = ceil_div(o.OW, t.nc), units = o.CB * 8 * ncg * ceil_div(o.OH, t.r);
        if (units > kThreads) continue;
        const int cost = ((t.r - 1) * t.s + 3) * ((t.nc - 1) * t.s + (t.full ? 1 : 3)) * 5 + t.r * t.nc * 40;
        if (o.tile < 0 || cost < best) { best = cost; o.tile = i; o.ncg = ncg; o.units = units; }
    }
    if (o.tile < 0) return false;
    // orientation: cycles of a K step; an MMA takes the larger of (128 + N) / 4 (operand reads) and N / 2
    auto mma = [](int n) { return n / 2 > (128 + n) / 4 ? n / 2 : (128 + n) / 4; };
    const int Kp = o.KB * 32, tiles = ceil_div(Kp, 128);
    o.wide = x3 && 2 * o.pxp <= 256 ? 1 : 0;
    const int on_m = tiles * (!x3 ? mma(o.pxp) : o.wide ? mma(2 * o.pxp) + mma(o.pxp) : 3 * mma(o.pxp));
    const int on_n = x3 ? mma(2 * Kp) + mma(Kp) : mma(Kp);
    // (pixels on M only where the tensor-memory lanes are mostly real: the epilogue's threads are pixels then)
    o.pix_m = o.px > 64 && o.px <= 128 && Kp <= 64 && on_n <= on_m ? 1 : 0;
    if (o.pix_m) o.wide = 0;
    o.m_tiles = o.pix_m ? 1 : tiles;
    o.rows = Kp < 128 ? Kp : 128;
    o.d_cols = (uint32_t)(o.pix_m ? (x3 ? 2 * Kp : Kp) : o.wide ? 2 * o.pxp : o.pxp);
    auto idesc = [](int n) { return (1u << 4) | (2u << 7) | (2u << 10) | ((uint32_t)(n >> 3) << 17) | ((128u >> 4) << 24); };
    o.idesc = idesc(o.pix_m ? Kp : o.pxp);
    o.idesc_wide = idesc(o.pix_m ? (x3 ? 2 * Kp : Kp) : o.wide ? 2 * o.pxp : o.pxp);
    o.in_stride = round_up((uint32_t)(o.H * o.W) * kPitch, 128);
    o.op_stride = (uint32_t)o.pxp * 128u * (x3 ? 2u : 1u);
    o.out_stride = round_up((uint32_t)o.px * kPitch, 128);
    o.dw_relu = (A.flags & SMALL_RELU) ? 1 : 0; o.relu = (Bn.flags & SMALL_RELU) ? 1 : 0;
    o.dw_w = A.w_blk; o.dw_bias = A.bias; o.bias = Bn.bias;
    return true;
}

// Structure of the list: does layer i start a pair of the run, reading slot `src` (any, where the run starts)?  Not where the 1x1 layer
// called on its own computes in FP32 (few products per pixel): its results stay FP32's.
bool is_pair(small_ctx *ctx, const small_layer *layers, int n, int i, int N, unsigned &math) {
    if (i + 1 >= n) return false;
    const small_layer &A = layers[i], &Bn = layers[i + 1];
    if (A.op != SMALL_OP_DWCONV || Bn.op != SMALL_OP_CONV) return false;
    const unsigned m = Bn.flags & SMALL_MATH_MASK;
    if (m != SMALL_MATH_TF32 && m != SMALL_MATH_3XTF32) return false;
    if (math == ~0u) math = m;
    if (m != math || A.FH != 3 || A.FW != 3 || A.stride < 1 || A.stride > 2) return false;
    if (Bn.FH != 1 || Bn.FW != 1 || Bn.stride != 1 || (Bn.pad_t | Bn.pad_b | Bn.pad_l | Bn.pad_r) || (Bn.flags & SMALL_ACCUMULATE)) return false;
    Geom g, gp;
    if (make_geom(g, N, A.C, A.C, A.H, A.W, 3, 3, A.stride, A.pad_t, A.pad_b, A.pad_l, A.pad_r)) return false;
    return A.dst >= 0 && Bn.src == A.dst && Bn.dst != A.dst && Bn.C == A.C && Bn.H == g.OH && Bn.W == g.OW &&
           make_geom(gp, N, A.C, Bn.K, g.OH, g.OW, 1, 1, 1, 0, 0, 0, 0) == SMALL_OK && slot_dead_after(layers, n, i + 2, A.dst) && !conv_in_fp32(ctx, gp, m);
}

// The longest run at layer i (pairs = 0: none).  Results that fit are in p.
void plan_run(small_ctx *ctx, const small_layer *layers, int n, int i, int N, Plan &p) {
    const size_t max_smem = ctx->max_smem_optin;
    const int sms = ctx->sm_count;
    p = Plan{};
    unsigned math = ~0u;
    Args &a = p.a;
    std::vector<int> ends;                               // structure: pairs that could follow one another
    int at = i;
    while ((int)ends.size() < kMaxPairs && is_pair(ctx, layers, n, at, N, math)) {
        if (at > i) {                                    // reads what the pair before it wrote, as its only reader
            const small_layer &P = layers[at - 1], &A = layers[at];
            if (A.src != P.dst || P.dst < 0 || A.C != P.K || A.H != P.H || A.W != P.W || !slot_dead_after(layers, n, at + 1, P.dst)) break;
        }
        ends.push_back(at);
        at += 2;
    }
    const bool x3 = math == SMALL_MATH_3XTF32;
    const int src = layers[i].src;
    for (int pairs = (int)ends.size(); pairs >= kMinPairs; --pairs) {
        const int end = i + 2 * pairs;
        // the head: a global average pool over the run's result and the full reduction behind it
        bool head = false;
        if (end + 1 < n) {
            const small_layer &P = layers[end - 1], &L = layers[end], &F = layers[end + 1];
            head = L.op == SMALL_OP_POOL && F.op == SMALL_OP_FC && L.src == P.dst && P.dst >= 0 && L.pool_mode == SMALL_POOL_AVG && L.C == P.K && L.H == P.H &&
                   L.W == P.W && L.FH == L.H && L.FW == L.W && !(L.pad_t | L.pad_b | L.pad_l | L.pad_r) && L.dst >= 0 && F.src == L.dst && F.dst != L.dst &&
                   F.C == L.C && F.K >= 1 && F.K <= 1024 && slot_dead_after(layers, n, end + 1, P.dst) && slot_dead_after(layers, n, end + 2, L.dst) &&
                   F.dst != src && small_gap_fc_fused(N, F.C, F.K, F.flags & SMALL_MATH_MASK);
        }
        if (!head && layers[end - 1].dst == src) continue;       // an image's result must not land where another's input is still to be read
        // two blocks on an SM where there are images for them and both fit
        for (p.per_sm = N > sms ? 2 : 1; p.per_sm; --p.per_sm) {
            a = Args{};
            bool ok = true;
            uint32_t plane = 0, stage = 0, cols = 32, floats = 0, needs[kMaxPairs];
            int blocks = 1;
            for (int j = 0; j < pairs && ok; ++j) {
                PairOp &o = a.p[j];
                ok = plan_pair(layers[i + 2 * j], layers[i + 2 * j + 1], N, x3, p.per_sm == 2 ? kTilesTwo : kTileCount, o);
                if (!ok) break;
                needs[j] = 0;
                auto need = [&](uint32_t bytes) { if (bytes > needs[j]) needs[j] = bytes; };
                need((uint32_t)o.CB * o.in_stride);
                need((uint32_t)(o.CB - 1) * o.op_stride + (o.pix_m ? (x3 ? (uint32_t)o.pxp : 0u) * 128u + 128u * 128u : o.op_stride));
                need((uint32_t)o.KB * o.out_stride);
                if (needs[j] > plane) plane = needs[j];
                const uint32_t box = (uint32_t)o.rows * 128u * (x3 ? 2u : 1u);
                if (box > stage) stage = box;
                while (cols < o.m_tiles * o.d_cols + (o.pix_m ? 0u : 32u)) cols *= 2;
                if (o.CB > blocks) blocks = o.CB;
                o.dwb_at = (int)floats; floats += (uint32_t)o.CB * 32u;
                o.b_at = (int)floats; floats += (uint32_t)o.KB * 32u;
            }
            if (!ok) continue;
            plane = round_up(plane, 1024);
            // an MMA with filters on M reads 128 rows from either part of a box; what lies behind the ring is the plane
            if (plane < 16384u) plane = 16384u;
            a.head_b_at = (int)floats;
            if (head) floats += (uint32_t)blocks_of(layers[end + 1].K) * 32u;
            a.dww_bytes = (uint32_t)blocks * 1152u;
            const uint32_t tail = 2u * a.dww_bytes + floats * 4u + 1280u * 4u + 16u * kMaxRing + 128u;
            auto total = [&](int ring) { return 1024u + (uint32_t)ring * stage + plane + tail; };
            // (each block and the SM reserve 1 KB)
            const uint32_t room = p.per_sm == 2 ? (uint32_t)((max_smem + 1024) / 2 - 1024) : (uint32_t)max_smem;
            if (cols > (p.per_sm == 2 ? 256u : 512u)) continue;
            if (total(2) > room) continue;
            a.ring = 2;
            while (a.ring < kMaxRing && total(a.ring + 1) <= room) ++a.ring;
            a.n = pairs; a.N = N;
            a.stage_bytes = stage; a.tmem_cols = (int)cols;
            a.plane_off = (uint32_t)a.ring * stage;
            a.dww_off = a.plane_off + plane;
            a.bias_off = a.dww_off + 2u * a.dww_bytes;
            a.head_off = a.bias_off + floats * 4u;
            a.ctrl_off = a.head_off + 1280u * 4u;
            if (N <= sms)                                    // one image per block: stages in what the later layers leave of the plane
                for (int g = 1; g < pairs && !a.grow_at; ++g) {
                    uint32_t left = 1024;
                    bool whole = true;                       // (an MMA with filters on M reads 128 rows)
                    for (int j = g; j < pairs; ++j) {
                        left = needs[j] > left ? needs[j] : left;
                        whole = whole && (a.p[j].pix_m || a.p[j].rows == 128);
                    }
                    left = round_up(left, 1024);
                    const int extra = left < plane && whole ? (int)((plane - left) / stage) : 0;
                    if (extra < 1 || a.ring == kMaxRing) continue;
                    a.grow_at = g;
                    a.ring2 = a.ring + extra < kMaxRing ? a.ring + extra : kMaxRing;
                    a.extra_off = a.plane_off + left;
                }
            // Every image streams the filters through its block.  With a block for every image that is hidden; with several rounds of
            // images the layer kernels, which read them once per tile of many images, win where there are many filters and few pixels
            // (us, layer by layer / as a run, 3xTF32: 64 channels on 25 x 5 batch 1000 140 / 78, on 12 x 12 162 / 147; 128 on 6 x 6 batch 148
            // 63 / 26, 400 81 / 64, 1000 121 / 139; 256 on 6 x 6 148 58 / 33, 400 98 / 86 but TF32 71 / 78; 256 on 3 x 3 148 46 / 27, 400 55 / 70).
            long long products = 0, pixels = 0;
            for (int j = 0; j < pairs; ++j) { products += (long long)a.p[j].C * a.p[j].K; pixels += a.p[j].px; }
            const int rounds = ceil_div(N, sms * p.per_sm);
            if (rounds > 1 && products > (rounds <= 3 ? 500 : 100) * pixels) continue;
            p.smem = total(a.ring);
            p.pairs = pairs; p.layers = 2 * pairs + (head ? 2 : 0); p.math = math;
            if (head) {
                const small_layer &F = layers[end + 1];
                a.head_w = F.w_blk; a.head_bias = F.bias; a.head_K = F.K; a.head_relu = (F.flags & SMALL_RELU) ? 1 : 0;
            }
            return;
        }
    }
    p.pairs = p.layers = 0;
}

struct Launch { const float *in; float *out; Maps maps; };
struct Entry { std::vector<unsigned char> key; std::unique_ptr<Plan> p; std::vector<Launch> made; };
typedef std::unordered_multimap<size_t, Entry> State;

// The finished plan for a list, a layer of it and a batch, made once (every call of a network asks).
Entry &entry_of(small_ctx *ctx, const small_layer *layers, int n, int i, int N) {
    if (!ctx->chain_state) ctx->chain_state = new State();
    State &s = *static_cast<State *>(ctx->chain_state);
    const int head[3] = {N, i, n};
    const size_t lb = sizeof(small_layer) * (size_t)(n - i);
    const size_t words = (((size_t)N * 64 + i) * 64 + n) ^ (reinterpret_cast<size_t>(layers[i].w_blk) << 16) ^ (reinterpret_cast<size_t>(layers[n - 1].w_blk) << 20);
    const auto range = s.equal_range(words);
    for (auto it = range.first; it != range.second; ++it) {
        Entry &e = it->second;
        if (e.key.size() == lb + sizeof(head) && !memcmp(e.key.data(), head, sizeof(head)) && !memcmp(e.key.data() + sizeof(head), layers + i, lb)) return e;
    }
    Entry e;
    e.key.resize(lb + sizeof(head));
    memcpy(e.key.data(), head, sizeof(head));
    memcpy(e.key.data() + sizeof(head), layers + i, lb);
    Plan p;
    plan_run(ctx, layers, n, i, N, p);
    if (p.layers) e.p.reset(new Plan(p));
    if (s.size() >= 512) s.clear();
    return s.emplace(words, std::move(e))->second;
}

}  // namespace

void free_chain_state(small_ctx *ctx) {
    delete static_cast<State *>(ctx->chain_state);
    ctx->chain_state = nullptr;
}

int sep_chain_layers(small_ctx *ctx, const small_layer *layers, int n, int i, int N) {
    if (n - i < 2 * kMinPairs || layers[i].op != SMALL_OP_DWCONV || layers[i + 1].op != SMALL_OP_CONV || layers[i + 2].op != SMALL_OP_DWCONV) return 0;
    const Plan *p = entry_of(ctx, layers, n, i, N).p.get();
    return p ? p->layers : 0;
}

int launch_sep_chain(small_ctx *ctx, const small_layer *layers, int n, int i, int N, const float *in, float *out, cudaStream_t st) {
    Entry &e = entry_of(ctx, layers, n, i, N);
    if (!e.p) return SMALL_ERR_UNSUPPORTED;
    const bool x3 = e.p->math == SMALL_MATH_3XTF32;
    const Launch *made = nullptr;
    for (const Launch &l : e.made)
        if (l.in == in && l.out == out) made = &l;
    if (!made) {
        EncodeTiledFn encode = reinterpret_cast<EncodeTiledFn>(ctx->encode_tiled);
        Launch l{};
        l.in = in; l.out = out;
        const Args &a = e.p->a;
        auto check = [&](CUresult r) { if (r != CUDA_SUCCESS) ctx->last_cuda = (int)r; return r == CUDA_SUCCESS; };
        {
            const PairOp &o = a.p[0];
            cuuint64_t dims[5] = {32, (cuuint64_t)o.W, (cuuint64_t)o.H, (cuuint64_t)o.CB, (cuuint64_t)N};
            cuuint64_t strides[4] = {128, (cuuint64_t)o.W * 128, (cuuint64_t)o.H * o.W * 128, (cuuint64_t)o.CB * o.H * o.W * 128};
            cuuint32_t box[5] = {kPitch / 4, (cuuint32_t)o.W, (cuuint32_t)o.H, 1, 1}, es[5] = {1, 1, 1, 1, 1};
            if (!check(encode(&l.maps.in, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 5, const_cast<float *>(in), dims, strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE,
                              CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE))) return SMALL_ERR_CUDA;
        }
        for (int j = 0; j < a.n; ++j) {
            const PairOp &o = a.p[j];
            const small_layer &L = layers[i + 2 * j + 1];
            const float *w[2];
            w[0] = L.w_blk + conv_w_fp32_elems(L.C, L.K, 1, 1);
            w[1] = x3 ? w[0] + conv_w_tc_elems(L.C, L.K, 1, 1) : w[0];
            for (int h = 0; h < 2; ++h) {      // [CB][KB * 32][32]
                cuuint64_t dims[3] = {32, (cuuint64_t)o.KB * 32, (cuuint64_t)o.CB}, strides[2] = {128, (cuuint64_t)o.KB * 32 * 128};
                cuuint32_t box[3] = {32, (cuuint32_t)o.rows, 1}, es[3] = {1, 1, 1};
                if (!check(encode(&l.maps.w[j][h], CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3, const_cast<float *>(w[h]), dims, strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE,
                                  CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE))) return SMALL_ERR_CUDA;
            }
        }
        if (e.made.size() >= 64) e.made.clear();
        e.made.push_back(l);
        made = &e.made.back();
    }
    Args a = e.p->a;
    a.out = out; a.status = ctx->dev_status; a.wait_iters = ctx->wait_iters; a.late = ctx->dependent == 2;
    const bool two = e.p->per_sm == 2;
    auto kern = x3 ? (two ? sep_chain_kernel<true, 2> : sep_chain_kernel<true, 1>) : (two ? sep_chain_kernel<false, 2> : sep_chain_kernel<false, 1>);
    cudaError_t err = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)ctx->max_smem_optin);
    if (err != cudaSuccess) { ctx->last_cuda = (int)err; return SMALL_ERR_CUDA; }
    const int most = ctx->sm_count * e.p->per_sm;
    launch_kernel(ctx, kern, dim3((unsigned)(N < most ? N : most)), dim3(kThreads), e.p->smem, st, made->maps, a);
    return check_launch(ctx);
}

}  // namespace small
