// A run of layers of a network as ONE kernel, one image at a time in shared memory (paper Section 6, the abstract fused
// layer, taken to whole stages: Section 5.3's layers share buffers, here the buffers never leave the SM).
//
// Why.  The networks the paper evaluates are tiny - a layer of one image is a few hundred thousand multiply-adds on a
// plane of at most a few thousand pixels - so launched layer by layer they spend their time filling and draining 148 SMs
// ten to thirty times: a launch takes 4 to 13 us whatever the batch, most of it start-up, the first copy's latency, and
// the last tile.  A layer here ends with a barrier of one thread block, or of the few that share an image.
//
// Work split.  A cluster of G thread blocks (1, 2, 4 or 8: as many as the batch leaves SMs for) takes one image after the
// other.  Every block of a cluster holds ALL activations of the image; it computes its share of a convolution's output
// (filters split over the blocks, then pixels) and stores each value into every block's copy (distributed shared memory),
// then a cluster barrier.  Depthwise layers are cheap and computed by every block for itself: no exchange.
//
// Layout of an activation: [pixel][pitch] floats, pitch = channels rounded up to 8, plus 4: the 16-byte chunks that eight
// consecutive pixels hold at one channel then lie in eight different bank groups for every channel count, so ldmatrix and
// 16-byte accesses are conflict-free without a swizzle.  Taps outside the plane read a zero area instead.
//
// Arithmetic.  Tensor-core modes: warp-level m16n8k8 TF32 MMAs (see conv_mma.cu), activations by ldmatrix.  FP32 mode: a lane
// per filter, pixels in registers, FMAs.  The filters of all operations form one stream of chunks (12 KB, rows of one
// input channel and tap) that cp.async brings through a ring in shared memory from the packed FP32 section, across the
// operations' ends: filters need no waiting for activations.  (Read straight from global memory by the warps that use them,
// with the next tap's in flight, every tap cost some 1500 cycles of latency.)  They are rounded to TF32 or split for 3xTF32 in
// registers.  A row's pitch of 40, 24 or 8 floats (32, 16 or 8 filters) makes the fragment reads conflict-free.
#pragma once

#include "common.cuh"
#include "sm100.cuh"

namespace small {
namespace resident {

constexpr int kMaxOps = 32, kMaxInputs = 4;
constexpr int kThreads = 512, kWarps = kThreads / 32;
constexpr int kZeroFloats = 32;             // what taps outside the plane read
constexpr int kScratchFloats = 4096;        // partial sums: K slices of a convolution, the pooling, the full reduction
constexpr int kMaxSteps = 512;              // K steps of a convolution
constexpr int kStages = 3, kStageFloats = 3072;

enum { kConv = 0, kDw = 1, kGap = 2, kFc = 3 };

struct alignas(16) Op {
    int kind;
    int C, K, H, W, OH, OW, FH, FW, S, pt, pl;
    int src, dst, sp, dp;                   // offsets (floats) of the tensors in shared memory, pitches
    int relu, accumulate;
    int exchange;                           // depthwise: the blocks of a cluster meet behind this operation
    int mf, nf, m_units, n_units;           // a warp's tile (fragments; FP32: nf = filters per lane), tiles of a block's part
    int lg_parts, n_parts, n_w, pitch, panel; // parts the filters are split into over the cluster, filters of a part, row pitch, floats of a panel in a stage
    int rows, chunk_rows, chunks;           // filter rows (multiples of 8), rows per chunk, chunks per pass over the filters
    int rounds;                             // passes: a warp computes one tile per pass
    int lg_split, split;                    // warps that share a tile's K steps
    int segs, seg_rows;                     // depthwise: runs of rows a column is cut into, rows of a run
    uint32_t by_ow, by_units, by_c4, by_cols;   // divisors as multipliers (see quotient): OW, n_units, channel quads, depthwise columns
    const float *w, *bias;
};
struct Input { const float *g; int C, H, W, off, pitch; };
struct Args {
    Op op[kMaxOps];
    Input in[kMaxInputs];
    int n_ops, n_stream, n_in, N, G;        // n_stream: operations with streamed filters (all but the head)
    int zero, scratch, ring, steps, ops;    // offsets (floats)
    float *out;                             // the full reduction's result, blocked [N][KB][1][1][32]
};

typedef void (*Kernel)(const Args);
Kernel resident_kernel_fp32();              // one translation unit each (net_resident_inst_*.cu)
Kernel resident_kernel_tf32();
Kernel resident_kernel_x3();

#ifdef SMALL_RESIDENT_KERNEL

__device__ __forceinline__ void cluster_sync() {
    asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
}
__device__ __forceinline__ uint32_t map_rank(uint32_t addr, uint32_t rank) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
    return r;
}
__device__ __forceinline__ void st_cluster4(uint32_t addr, const float (&v)[4]) {
    asm volatile("st.shared::cluster.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "f"(v[0]), "f"(v[1]), "f"(v[2]), "f"(v[3]) : "memory");
}
__device__ __forceinline__ void st_cluster1(uint32_t addr, float x) {
    asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(addr), "f"(x) : "memory");
}
__device__ __forceinline__ void ldsm4(uint32_t addr, uint32_t (&r)[4]) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}
__device__ __forceinline__ void mma_16x8x8(float (&c)[4], const uint32_t *a, const uint32_t *b) {
    asm("mma.sync.aligned.m16n8k8.row.col.f32.tf32.tf32.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3]) : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}
__device__ __forceinline__ void cp16(uint32_t dst, const void *src, int bytes) {      // bytes < 16: the rest is zero
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(bytes) : "memory");
}

__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {      // two FMAs
    uint64_t r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
// n / d by a multiplication: m = 2^32 / d + 1, 0 for d = 1; exact for n * d < 2^32
__device__ __forceinline__ int quotient(int n, uint32_t m) { return m ? (int)__umulhi((uint32_t)n, m) : n; }

// bit t: tap t = x * FW + y of the window at (ih0, iw0) lies inside the plane (at most 25 taps)
__device__ __forceinline__ uint32_t tap_mask(const Op &o, int ih0, int iw0) {
    if (o.FH == 1 && o.FW == 1) return (unsigned)ih0 < (unsigned)o.H && (unsigned)iw0 < (unsigned)o.W ? 1u : 0u;
    const int y0 = max(0, -iw0), y1 = min(o.FW, o.W - iw0);
    const uint32_t row = y1 > y0 ? ((1u << y1) - 1u) & ~((1u << y0) - 1u) : 0u;
    uint32_t m = 0;
#pragma unroll 1
    for (int x = max(0, -ih0); x < min(o.FH, o.H - ih0); ++x) m |= row << (x * o.FW);
    return m;
}

// The stream of filter chunks: (op, round, chunk) is the next one to be copied, `put` and `get` count stages.
struct Stream {
    int op, round, chunk, put, get, left;                // left: images whose filters are still to be streamed
};

// Copies the next chunk into its stage (one commit group per call, empty at the end).
__device__ __forceinline__ void stream_issue(const Args &a, const Op *ops, Stream &st, const uint32_t sm, const int rank) {
    if (st.left > 0) {
        const Op &o = ops[st.op];
        const uint32_t dst = sm + (uint32_t)(a.ring + st.put * kStageFloats) * 4u;
        const int CB = (o.C + 31) >> 5;
        if (o.kind == kDw) {
            const int nw = CB * 72;                                                // 16-byte pieces of the filters, then of the bias
#pragma unroll 1
            for (int i = threadIdx.x; i < nw + CB * 8; i += kThreads) {
                const int left = o.bias ? o.C - (i - nw) * 4 : 0;
                cp16(dst + i * 16, i < nw ? o.w + i * 4 : left > 0 ? o.bias + (i - nw) * 4 : o.w, i < nw || left >= 4 ? 16 : left > 0 ? left * 4 : 0);
            }
        } else {
            const int T = o.FH * o.FW, tail = (o.C - (CB - 1) * 32 + 7) & ~7, main = (CB - 1) * T * 32;
            const int r0 = st.chunk * o.chunk_rows, nr = min(o.chunk_rows, o.rows - r0);
            const int k0 = (rank & (o.n_parts - 1)) * o.n_w, inv = 65536 / tail + 1;
            const int pw4 = min(o.n_w, 32) >> 2, sh = pw4 == 8 ? 3 : pw4 == 4 ? 2 : 1;      // 16-byte pieces of a panel's row
            const int q = threadIdx.x & (pw4 - 1);
#pragma unroll 1
            for (int pn = 0; pn * 32 < o.n_w; ++pn) {
                const int k = k0 + pn * 32;
                const float *w = o.w + (size_t)(k >> 5) * CB * T * 1024 + (k & 31) + q * 4;
                const uint32_t d = dst + (uint32_t)(pn * o.panel + q * 4) * 4u;
#pragma unroll 1
                for (int j = threadIdx.x >> sh; j < nr; j += kThreads >> sh) {
                    const int g = r0 + j, g2 = g - main, t = (g2 * inv) >> 16;
                    cp16(d + (uint32_t)(j * o.pitch) * 4u, w + (g2 < 0 ? g * 32 : main * 32 + t * 1024 + (g2 - t * tail) * 32), 16);
                }
            }
        }
        if (++st.put == kStages) st.put = 0;
        if (o.kind == kDw || (++st.chunk == o.chunks && (st.chunk = 0, ++st.round) == o.rounds)) {
            st.round = 0;
            if (++st.op == a.n_stream) { st.op = 0; --st.left; }
        }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
}
// The chunk in turn is in place for every thread (and everything before this in the block is done); the stage behind goes
// back into the stream.  Returns its place in shared memory.
__device__ __forceinline__ int stream_next(const Args &a, const Op *ops, Stream &st, const uint32_t sm, const int rank) {
    asm volatile("cp.async.wait_group %0;" ::"n"(kStages - 2) : "memory");
    __syncthreads();
    const int at = a.ring + st.get * kStageFloats;
    if (++st.get == kStages) st.get = 0;
    stream_issue(a, ops, st, sm, rank);
    return at;
}

// The K steps (8 channels of a tap) of an operation: byte offset of the step from a pixel's first tap, and the tap.
__device__ __forceinline__ void fill_steps(const Op &o, int *tab) {
    const int T = o.FH * o.FW, CB = (o.C + 31) >> 5, main = (CB - 1) * T * 4, tail = (o.C - (CB - 1) * 32 + 7) >> 3;
#pragma unroll 1
    for (int i = threadIdx.x; i < (o.rows >> 3); i += kThreads) {
        const bool m = i < main;
        const int tl = m ? i >> 2 : (i - main) / tail, ks = m ? i & 3 : i - main - tl * tail;
        const int cb = m ? tl / T : CB - 1, tap = m ? tl - cb * T : tl, x = tap / o.FW, y = tap - x * o.FW;
        tab[i] = (tap << 24) | (((x * o.W + y) * o.sp + cb * 32 + ks * 8) * 4);
    }
}

// One chunk's K steps, every `split`-th, of a warp's tile on the tensor cores: MF fragments of 16 pixels x NF fragments of 8
// filters.  The next step's filters and table entry are in flight during a step (what they read past a chunk is not used).
template <bool X3, int MF, int NF>
__device__ __forceinline__ void mma_steps(float (&acc)[2][2][4], float (&accs)[2][2][4], const uint32_t (&base)[2], const uint32_t (&mask)[2], const uint32_t zero,
                                          const int *tab, const float *wp, const int pitch, const int steps, const int split) {
    float w[NF][2];
#pragma unroll
    for (int n = 0; n < NF; ++n) { w[n][0] = wp[n * 8]; w[n][1] = wp[4 * pitch + n * 8]; }
    int e = *tab;
#pragma unroll 1
    for (int i = 0; i < steps; i += split) {
        uint32_t av[MF][4];
#pragma unroll
        for (int m = 0; m < MF; ++m) ldsm4((mask[m] >> (e >> 24) & 1u) ? base[m] + (uint32_t)(e & 0xffffff) : zero, av[m]);
        uint32_t bh[NF][2], bl[NF][2];
#pragma unroll
        for (int n = 0; n < NF; ++n)
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                if (X3) {
                    bh[n][h] = __float_as_uint(w[n][h]) & 0xffffe000u;
                    bl[n][h] = __float_as_uint(w[n][h] - __uint_as_float(bh[n][h]));
                } else {
                    asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(bh[n][h]) : "f"(w[n][h]));
                }
            }
        tab += split;
        wp += 8 * pitch * split;
        e = *tab;
#pragma unroll
        for (int n = 0; n < NF; ++n) { w[n][0] = wp[n * 8]; w[n][1] = wp[4 * pitch + n * 8]; }
#pragma unroll
        for (int m = 0; m < MF; ++m) {
            if (X3) {
                uint32_t al[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const uint32_t h = av[m][j] & 0xffffe000u;
                    al[j] = __float_as_uint(__uint_as_float(av[m][j]) - __uint_as_float(h));
                    av[m][j] = h;
                }
#pragma unroll
                for (int n = 0; n < NF; ++n) {                      // the small products apart (shorter chains)
                    mma_16x8x8(accs[m][n], al, bh[n]);
                    mma_16x8x8(acc[m][n], av[m], bh[n]);
                    mma_16x8x8(accs[m][n], av[m], bl[n]);
                }
            } else {
#pragma unroll
                for (int n = 0; n < NF; ++n) mma_16x8x8(acc[m][n], av[m], bh[n]);
            }
        }
    }
}

// A block's part of a convolution on the tensor cores.  Every warp computes one tile per round, or every `split`-th K step of
// one where there are fewer tiles than warps.  The code is kept short on purpose (one copy of everything but the K steps,
// loops not unrolled): each operation runs through it once, and its instruction fetches were most of its time before.
template <bool X3>
__device__ __forceinline__ void conv_mma(const Args &a, const Op *ops, const Op &o, Stream &st, const uint32_t sm, float *smem, const int rank, int *tab) {
    const int lane = threadIdx.x & 31, warp = sm100::warp_index(), G = a.G;
    const int P = o.OH * o.OW, mf = o.mf, nf = o.nf;
    const int np = rank & (o.n_parts - 1), mp = rank >> o.lg_parts, m_parts = G >> o.lg_parts;
    const int slice = warp & (o.split - 1);
    const uint32_t chunk16 = (uint32_t)(lane >> 4) << 4, zero = sm + (uint32_t)a.zero * 4u;
    fill_steps(o, tab);
#pragma unroll 1
    for (int round = 0; round < o.rounds; ++round) {
        const int u = (round * kWarps + warp) >> o.lg_split, mu = quotient(u, o.by_units), nu = u - mu * o.n_units;
        const bool mine = mu < o.m_units;
        const int px0 = (mu * m_parts + mp) * mf * 16, n0 = nu * nf;               // first pixel of the layer, first filter fragment of the part
        uint32_t base[2], mask[2];
        float acc[2][2][4], accs[2][2][4], bias[2][4];
        const int k4 = np * o.n_w + n0 * 8 + ((lane & 2) << 1);                    // first of the four filters this lane stores of a fragment
        if (mine)
#pragma unroll
        for (int m = 0; m < 2; ++m) {
            // this lane's row of the A fragments: pixel lane & 15, 16-byte chunk lane >> 4 of a K step
            const int px = px0 + m * 16 + (lane & 15), oh = quotient(px, o.by_ow), ow = px - oh * o.OW;
            const int ih0 = oh * o.S - o.pt, iw0 = ow * o.S - o.pl;
            base[m] = sm + (uint32_t)((o.src + (ih0 * o.W + iw0) * o.sp) * 4) + chunk16;
            mask[m] = px < P && m < mf ? tap_mask(o, ih0, iw0) : 0u;
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int k = k4 + m * 8 + j;
                bias[m][j] = o.bias && m < nf && k < o.K ? __ldg(o.bias + k) : 0.0f;
            }
        }
#pragma unroll
        for (int m = 0; m < 2; ++m)
#pragma unroll
            for (int n = 0; n < 2; ++n)
#pragma unroll
                for (int e = 0; e < 4; ++e) acc[m][n][e] = accs[m][n][e] = 0.0f;
#pragma unroll 1
        for (int c = 0; c < o.chunks; ++c) {
            const int at = stream_next(a, ops, st, sm, rank);
            if (!mine) continue;
            const int steps = (min(o.chunk_rows, o.rows - c * o.chunk_rows) >> 3) - slice;
            const float *wp = smem + at + (n0 >> 2) * o.panel + ((lane & 3) + 8 * slice) * o.pitch + (n0 & 3) * 8 + (lane >> 2);
            const int *tp = tab + c * (o.chunk_rows >> 3) + slice;
            if (nf == 1) mma_steps<X3, 1, 1>(acc, accs, base, mask, zero, tp, wp, o.pitch, steps, o.split);
            else if (mf == 1) mma_steps<X3, 1, 2>(acc, accs, base, mask, zero, tp, wp, o.pitch, steps, o.split);
            else mma_steps<X3, 2, 2>(acc, accs, base, mask, zero, tp, wp, o.pitch, steps, o.split);
        }
        if (X3)
#pragma unroll
            for (int m = 0; m < 2; ++m)
#pragma unroll
                for (int n = 0; n < 2; ++n)
#pragma unroll
                    for (int e = 0; e < 4; ++e) acc[m][n][e] += accs[m][n][e];
        if (o.split > 1) {                               // the slices of a tile add up in the first one's registers
            float *part = smem + a.scratch + (u * (o.split - 1) + slice - 1) * mf * nf * 128 + lane;
            if (slice && mine)
#pragma unroll
                for (int m = 0; m < 2; ++m)
#pragma unroll
                    for (int n = 0; n < 2; ++n)
                        if (m < mf && n < nf)
#pragma unroll
                            for (int e = 0; e < 4; ++e) part[((m * nf + n) * 4 + e) * 32] = acc[m][n][e];
            __syncthreads();
            if (slice) continue;
#pragma unroll 1
            for (int s = 1; s < o.split; ++s) {
                part += mf * nf * 128;
#pragma unroll
                for (int m = 0; m < 2; ++m)
#pragma unroll
                    for (int n = 0; n < 2; ++n)
                        if (m < mf && n < nf && mine)
#pragma unroll
                            for (int e = 0; e < 4; ++e) acc[m][n][e] += part[((m * nf + n) * 4 + e) * 32];
            }
        }
        if (!mine) continue;
        // Neighbouring lanes exchange halves, so that each holds four filters of one pixel; + bias, + the tensor already in
        // place, ReLU; into every block's copy.
        const int Kp = (o.K + 7) & ~7, odd = lane & 1;
        uint32_t at[2][2];
#pragma unroll
        for (int m = 0; m < 2; ++m)
#pragma unroll
            for (int n = 0; n < 2; ++n) {
                float *v = acc[m][n];
                const float s0 = __shfl_xor_sync(0xffffffffu, odd ? v[0] : v[2], 1), s1 = __shfl_xor_sync(0xffffffffu, odd ? v[1] : v[3], 1);
                if (odd) { v[0] = s0; v[1] = s1; } else { v[2] = s0; v[3] = s1; }
                const int px = px0 + m * 16 + (lane >> 2) + 8 * odd, k = k4 + n * 8;
                const bool ok = m < mf && n < nf && px < P && k < Kp;
                const int to = o.dst + px * o.dp + k;
                at[m][n] = ok ? (uint32_t)to : 0xffffffffu;
                if (ok) {
                    float4 p = make_float4(0.f, 0.f, 0.f, 0.f);
                    if (o.accumulate) p = *reinterpret_cast<const float4 *>(smem + to);
                    v[0] += bias[n][0] + p.x; v[1] += bias[n][1] + p.y; v[2] += bias[n][2] + p.z; v[3] += bias[n][3] + p.w;
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        if (o.relu) v[j] = fmaxf(v[j], 0.0f);
                        if (k + j >= o.K) v[j] = 0.0f;
                    }
                }
            }
#pragma unroll 1
        for (int r = 0; r < G; ++r) {
            const uint32_t to = G > 1 ? map_rank(sm, (uint32_t)r) : 0u;
#pragma unroll
            for (int m = 0; m < 2; ++m)
#pragma unroll
                for (int n = 0; n < 2; ++n)
                    if (at[m][n] != 0xffffffffu) {
                        if (G > 1) st_cluster4(to + at[m][n] * 4u, acc[m][n]);
                        else *reinterpret_cast<float4 *>(smem + at[m][n]) = make_float4(acc[m][n][0], acc[m][n][1], acc[m][n][2], acc[m][n][3]);
                    }
        }
    }
}

// The same in FP32: a lane per filter (Q filters 32 apart), eight consecutive pixels in registers; with fewer than 32 filters
// (n_w = 16 or 8) the parts of a warp take different pixels.  Activations are 16-byte shared-memory broadcasts.
// (Two FMAs per instruction, even and odd channels apart, take 16 registers more and spill: 50 -> 55 us on the keyword-spotting net.)
template <int Q>
__device__ __forceinline__ void fma_steps(float (&acc)[8][2], const int (&base)[8], const uint32_t (&mask)[8], const int zero, const float *smem, const int *tab,
                                          const float *wp, const int panel, const int pitch, const int steps, const int split) {
#pragma unroll 1
    for (int i = 0; i < steps; i += split) {
        const int e = *tab, tap = e >> 24, off = (e & 0xffffff) >> 2;
        int at[8];
#pragma unroll
        for (int p = 0; p < 8; ++p) at[p] = (mask[p] >> tap & 1u) ? base[p] + off : zero;
#pragma unroll
        for (int c4 = 0; c4 < 2; ++c4) {
            float w[Q][4];
#pragma unroll
            for (int q = 0; q < Q; ++q)
#pragma unroll
                for (int j = 0; j < 4; ++j) w[q][j] = wp[q * panel + (c4 * 4 + j) * pitch];
#pragma unroll
            for (int p = 0; p < 8; ++p) {
                const float4 v = *reinterpret_cast<const float4 *>(smem + at[p] + c4 * 4);
#pragma unroll
                for (int q = 0; q < Q; ++q) acc[p][q] = fmaf(v.w, w[q][3], fmaf(v.z, w[q][2], fmaf(v.y, w[q][1], fmaf(v.x, w[q][0], acc[p][q]))));
            }
        }
        tab += split;
        wp += 8 * pitch * split;
    }
}
__device__ __forceinline__ void conv_fma(const Args &a, const Op *ops, const Op &o, Stream &st, const uint32_t sm, float *smem, const int rank, int *tab) {
    const int lane = threadIdx.x & 31, warp = sm100::warp_index(), G = a.G, nq = o.nf;
    const int P = o.OH * o.OW, KW = min(o.n_w, 32), kl = lane & (KW - 1), lg_kw = KW == 32 ? 5 : KW == 16 ? 4 : 3;
    const int np = rank & (o.n_parts - 1), mp = rank >> o.lg_parts, m_parts = G >> o.lg_parts;
    const int slice = warp & (o.split - 1);
    fill_steps(o, tab);
#pragma unroll 1
    for (int round = 0; round < o.rounds; ++round) {
        const int u = (round * kWarps + warp) >> o.lg_split, mu = quotient(u, o.by_units), nu = u - mu * o.n_units;
        const bool mine = mu < o.m_units;
        const int px0 = (((mu * m_parts + mp) << (5 - lg_kw)) + (lane >> lg_kw)) * 8, k0 = np * o.n_w + nu * nq * 32 + kl;
        int base[8];
        uint32_t mask[8];
        float acc[8][2], bias[2];
        if (mine) {
            int oh = quotient(px0, o.by_ow), ow = px0 - oh * o.OW;
#pragma unroll
            for (int p = 0; p < 8; ++p) {
                const int ih0 = oh * o.S - o.pt, iw0 = ow * o.S - o.pl;
                base[p] = o.src + (ih0 * o.W + iw0) * o.sp;
                mask[p] = px0 + p < P ? tap_mask(o, ih0, iw0) : 0u;
                if (++ow == o.OW) { ow = 0; ++oh; }
            }
        }
#pragma unroll
        for (int p = 0; p < 8; ++p) acc[p][0] = acc[p][1] = 0.0f;
#pragma unroll
        for (int q = 0; q < 2; ++q) bias[q] = mine && o.bias && q < nq && k0 + q * 32 < o.K ? __ldg(o.bias + k0 + q * 32) : 0.0f;
#pragma unroll 1
        for (int c = 0; c < o.chunks; ++c) {
            const int at = stream_next(a, ops, st, sm, rank);
            if (!mine) continue;
            const int steps = (min(o.chunk_rows, o.rows - c * o.chunk_rows) >> 3) - slice;
            const float *wp = smem + at + nu * nq * o.panel + 8 * slice * o.pitch + kl;
            const int *tp = tab + c * (o.chunk_rows >> 3) + slice;
            if (nq == 1) fma_steps<1>(acc, base, mask, a.zero, smem, tp, wp, o.panel, o.pitch, steps, o.split);
            else fma_steps<2>(acc, base, mask, a.zero, smem, tp, wp, o.panel, o.pitch, steps, o.split);
        }
        if (o.split > 1) {                               // the slices of a tile add up in the first one's registers
            float *part = smem + a.scratch + (u * (o.split - 1) + slice - 1) * nq * 256 + lane;
            if (slice && mine)
#pragma unroll
                for (int q = 0; q < 2; ++q)
                    if (q < nq)
#pragma unroll
                        for (int p = 0; p < 8; ++p) part[(q * 8 + p) * 32] = acc[p][q];
            __syncthreads();
            if (slice) continue;
#pragma unroll 1
            for (int s = 1; s < o.split; ++s) {
                part += nq * 256;
#pragma unroll
                for (int q = 0; q < 2; ++q)
                    if (q < nq && mine)
#pragma unroll
                        for (int p = 0; p < 8; ++p) acc[p][q] += part[(q * 8 + p) * 32];
            }
        }
        if (!mine) continue;
        const int Kp = (o.K + 7) & ~7;
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const int k = k0 + q * 32;
            if (q >= nq || k >= Kp) continue;
            const int to0 = o.dst + px0 * o.dp + k, left = P - px0;
#pragma unroll
            for (int p = 0; p < 8; ++p) {
                float v = acc[p][q] + bias[q];
                if (o.accumulate && p < left) v += smem[to0 + p * o.dp];
                if (o.relu) v = fmaxf(v, 0.0f);
                acc[p][q] = k < o.K ? v : 0.0f;
            }
#pragma unroll 1
            for (int r = 0; r < G; ++r) {
                const uint32_t to = G > 1 ? map_rank(sm, (uint32_t)r) + (uint32_t)to0 * 4u : 0u;
#pragma unroll
                for (int p = 0; p < 8; ++p)
                    if (p < left) {
                        if (G > 1) st_cluster1(to + (uint32_t)(p * o.dp) * 4u, acc[p][q]);
                        else smem[to0 + p * o.dp] = acc[p][q];
                    }
            }
        }
    }
}

// Depthwise 3 x 3: a thread walks down a run of output rows of one column and four channels, the window in registers (two
// channels per FMA instruction).  Columns outside the plane read the zero area with a row step of nothing.
template <int S>
__device__ __forceinline__ void dw_layer(const Args &a, const Op &o, float *smem, const int wat) {
    const int C4 = ((o.C + 7) & ~7) >> 2, cols = o.OW * C4;
#pragma unroll 1
    for (int u = threadIdx.x; u < cols * o.segs; u += kThreads) {
        const int seg = quotient(u, o.by_cols), c = u - seg * cols, ow = quotient(c, o.by_c4), c4 = c - ow * C4;
        const int oh0 = seg * o.seg_rows, n = min(o.OH, oh0 + o.seg_rows) - oh0;
        const ulonglong2 *wt = reinterpret_cast<const ulonglong2 *>(smem + wat + (c4 >> 3) * 288) + (c4 & 7);
        ulonglong2 w[9];
#pragma unroll
        for (int i = 0; i < 9; ++i) w[i] = wt[i * 8];
        const ulonglong2 bias = reinterpret_cast<const ulonglong2 *>(smem + wat + ((o.C + 31) >> 5) * 288)[c4];
        const int iw0 = ow * S - o.pl, ih0 = oh0 * S - o.pt;
        const float *p[3];
        int step[3];
#pragma unroll
        for (int y = 0; y < 3; ++y) {
            const bool in = (unsigned)(iw0 + y) < (unsigned)o.W;
            p[y] = smem + (in ? o.src + (ih0 * o.W + iw0 + y) * o.sp + c4 * 4 : a.zero);
            step[y] = in ? o.W * o.sp : 0;
        }
        int ih = ih0;
        auto row = [&](ulonglong2 (&r)[3]) {
            const bool in = (unsigned)ih < (unsigned)o.H;
#pragma unroll
            for (int y = 0; y < 3; ++y) {
                r[y] = *reinterpret_cast<const ulonglong2 *>(in ? p[y] : smem + a.zero);
                p[y] += step[y];
            }
            ++ih;
        };
        ulonglong2 r0[3], r1[3], r2[3];
        row(r0);
        if (S == 1) row(r1);
        float *dst = smem + o.dst + (oh0 * o.OW + ow) * o.dp + c4 * 4;
#pragma unroll 1
        for (int i = 0; i < n; ++i, dst += o.OW * o.dp) {
            if (S == 2) row(r1);
            row(r2);
            ulonglong2 v = bias;
#pragma unroll
            for (int y = 0; y < 3; ++y) {
                v.x = fma2(r2[y].x, w[6 + y].x, fma2(r1[y].x, w[3 + y].x, fma2(r0[y].x, w[y].x, v.x)));
                v.y = fma2(r2[y].y, w[6 + y].y, fma2(r1[y].y, w[3 + y].y, fma2(r0[y].y, w[y].y, v.y)));
            }
            float4 f = make_float4(__uint_as_float((uint32_t)v.x), __uint_as_float((uint32_t)(v.x >> 32)), __uint_as_float((uint32_t)v.y), __uint_as_float((uint32_t)(v.y >> 32)));
            if (o.relu) { f.x = fmaxf(f.x, 0.f); f.y = fmaxf(f.y, 0.f); f.z = fmaxf(f.z, 0.f); f.w = fmaxf(f.w, 0.f); }
            *reinterpret_cast<float4 *>(dst) = f;
#pragma unroll
            for (int y = 0; y < 3; ++y) { if (S == 1) { r0[y] = r1[y]; r1[y] = r2[y]; } else r0[y] = r2[y]; }
        }
    }
}

// Global average pool: partial sums of pixel groups, then one sum per channel (four channels per thread throughout).
__device__ __forceinline__ void gap_layer(const Args &a, const Op &o, float *smem) {
    const int C4 = ((o.C + 7) & ~7) >> 2, P = o.H * o.W;
    const int groups = o.segs;
    const int g = quotient(threadIdx.x, o.by_c4), c4 = threadIdx.x - g * C4;
    float4 *part = reinterpret_cast<float4 *>(smem + a.scratch);
    if (g < groups) {
        float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 4
        for (int p = g; p < P; p += groups) {
            const float4 v = *reinterpret_cast<const float4 *>(smem + o.src + p * o.sp + c4 * 4);
            s.x += v.x; s.y += v.y; s.z += v.z; s.w += v.w;
        }
        part[g * C4 + c4] = s;
    }
    __syncthreads();
    if (threadIdx.x < C4) {
        float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 4
        for (int i = 0; i < groups; ++i) {
            const float4 v = part[i * C4 + c4];
            s.x += v.x; s.y += v.y; s.z += v.z; s.w += v.w;
        }
        const float n = (float)P;
        *reinterpret_cast<float4 *>(smem + o.dst + c4 * 4) = make_float4(s.x / n, s.y / n, s.z / n, s.w / n);
    }
}

// The full reduction behind it: a lane per filter, the channels shared out over the warps; straight to global memory.
__device__ __forceinline__ void fc_layer(const Args &a, const Op &o, float *smem, int n) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int KB = (o.K + 31) >> 5, CB = (o.C + 31) >> 5;
#pragma unroll 1
    for (int kb = 0; kb < KB; ++kb) {
        float s = 0.0f;
        const float *w = o.w + (size_t)kb * CB * 1024 + lane;
#pragma unroll 1
        for (int c0 = warp; c0 < o.C; c0 += 8 * kWarps) {           // eight rows in flight
            float v[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) v[i] = c0 + i * kWarps < o.C ? __ldg(w + (size_t)(c0 + i * kWarps) * 32) : 0.0f;
#pragma unroll
            for (int i = 0; i < 8; ++i) if (c0 + i * kWarps < o.C) s = fmaf(smem[o.src + c0 + i * kWarps], v[i], s);
        }
        smem[a.scratch + warp * 32 + lane] = s;
        __syncthreads();
        if (warp == 0) {
            const int k = kb * 32 + lane;
            float v = 0.0f;
#pragma unroll 4
            for (int i = 0; i < kWarps; ++i) v += smem[a.scratch + i * 32 + lane];
            if (k < o.K) { if (o.bias) v += __ldg(o.bias + k); if (o.relu) v = fmaxf(v, 0.0f); } else v = 0.0f;
            a.out[((size_t)n * KB + kb) * 32 + lane] = v;
        }
        __syncthreads();
    }
}

template <int MODE>      // 0: FP32, 1: TF32, 2: 3xTF32
__global__ void __launch_bounds__(kThreads, 1) net_resident_kernel(const __grid_constant__ Args a) {
    extern __shared__ __align__(16) float smem[];
    const uint32_t sm = sm100::smem_u32(smem);
    const int G = a.G;
    int rank = 0;
    if (G > 1) asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
    const int first = blockIdx.x / G, step = gridDim.x / G;
    Stream st{0, 0, 0, 0, 0, first < a.N ? (a.N - first + step - 1) / step : 0};
    Op *ops = reinterpret_cast<Op *>(smem + a.ops);
    for (int i = threadIdx.x; i < a.n_ops * (int)(sizeof(Op) / 4); i += kThreads) reinterpret_cast<int *>(ops)[i] = reinterpret_cast<const int *>(a.op)[i];
    __syncthreads();
#pragma unroll 1
    for (int i = 0; i < kStages - 1; ++i) stream_issue(a, ops, st, sm, rank);           // filters are no layer's output
    for (int i = threadIdx.x; i < kZeroFloats; i += kThreads) smem[a.zero + i] = 0.0f;
    grid_dep_sync();
    grid_dep_trigger();
    // (Runs are chosen so that every cluster has one image, see worth_it, and the loop turns once.  Written without it, the FP32
    // kernel's code comes out slower: keyword-spotting network, batch 75, 55.4 -> 57.4 us, and seven other ways no better.)
    for (int n = first; n < a.N; n += step) {
#pragma unroll 1
        for (int t = 0; t < a.n_in; ++t) {
            const Input &in = a.in[t];
            const int P = in.H * in.W, C4 = ((in.C + 7) & ~7) >> 2, CB = (in.C + 31) >> 5;
            const float4 *g = reinterpret_cast<const float4 *>(in.g) + (size_t)n * CB * P * 8;
#pragma unroll 4
            for (int i = threadIdx.x; i < P * C4; i += kThreads) {
                const int p = i / C4, c4 = i - p * C4;
                *reinterpret_cast<float4 *>(smem + in.off + p * in.pitch + c4 * 4) = g[((size_t)(c4 >> 3) * P + p) * 8 + (c4 & 7)];
            }
        }
        // the image's inputs are in place, and no block still works on the image before
        if (G > 1) cluster_sync(); else __syncthreads();
#pragma unroll 1
        for (int l = 0; l < a.n_ops; ++l) {
            const Op o = ops[l];                                    // in registers: fields read from the launch's constants where they are used cost a cache miss each
            if (o.kind == kConv) {
                int *tab = reinterpret_cast<int *>(smem) + a.steps + (l & 1) * kMaxSteps;      // (the operation before may still be reading its own)
                if constexpr (MODE == 0) conv_fma(a, ops, o, st, sm, smem, rank, tab);
                else conv_mma<MODE == 2>(a, ops, o, st, sm, smem, rank, tab);
                if (G > 1) cluster_sync();                          // one block: the next operation's first chunk is waited for by all
            } else if (o.kind == kDw) {
                const int wat = stream_next(a, ops, st, sm, rank);
                if (o.S == 1) dw_layer<1>(a, o, smem, wat); else dw_layer<2>(a, o, smem, wat);
                if (G > 1 && o.exchange) cluster_sync();
            } else if (rank == 0) {                                 // the classifier head: one block's work
                __syncthreads();
                if (o.kind == kGap) gap_layer(a, o, smem); else fc_layer(a, o, smem, n);
            }
        }
        __syncthreads();
    }
    if (G > 1) cluster_sync();                                      // no block leaves while another may still store into it
}

#endif  // SMALL_RESIDENT_KERNEL

}  // namespace resident
}  // namespace small
