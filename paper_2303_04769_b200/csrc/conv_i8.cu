// Quantised full channel reduction on the tensor cores (paper Section 3.2 item 4 on the uint8 tensors of Sections 5.1
// and 5.5; int32 accumulation as in Section 5.3): an implicit GEMM straight from the blocked uint8 layout with
// tcgen05.mma kind::i8, exact in every bit.
//
//   sum (x - zx)(w - zw) = sum x w  -  zw sum x  -  zx sum w  +  taps C zx zw          (all four modulo 2^32)
//
// sum x w is the MMA on the raw bytes.  sum x over a pixel's window comes out of the same MMA: behind the filters of a
// tile stands one more row of ones, so the accumulator has one more column.  The other two terms depend on the filter
// and on which taps of the window lie inside the plane: one constant per (border class of the pixel, filter), tabulated
// in shared memory by each thread block.  TMA's zero fill outside the plane adds nothing to the first two sums, which
// is the padding.
//
// Mapping: pixels on the MMA's M axis (128 consecutive pixels of a strip = a chunk), filters + the row of ones on N.  A
// pixel of a channel block is 32 bytes, exactly one K step of kind::i8, so a strip is [pixel][32 bytes] with the
// 32-byte swizzle and every window tap reads the same strip through a shifted start address, as in conv_tc.cu; stride 2
// is a stride-1 window over the input's four phase planes, read by TMA with element stride 2.
//
// Roles (640 threads, persistent): warp 0 loads strips, warp 2 filter boxes (resident for the whole kernel where they
// fit: a block keeps one filter tile and walks the pixel tiles), warp 1 issues the MMAs, warps 4-19 requantise and store.
// Two to eight accumulator slots, so the MMAs of the next tiles run beside the requantisation of the ones before them.
//
// What bounds it: the start.  Measured (batch 128, 64 -> 64 on 28 x 28, 3 x 3): 13.9 us, of which an empty layer takes 4.8; an SM
// has five or six chunks, 18 MMAs of 128 x 80 x 32 each ((128 + N) / 4 cycles of operand reads and some to issue, about 1200 cycles a
// chunk, 4 us in all), behind the arrival of all filters and the tables.  Tensor pipe 19 % of the active cycles, issue slots 45 %.
// The requantisation - per output one three-input add, one 64-bit multiply-add (rounding, bias and zero point in its addend), a
// shift, a maximum and half a saturating pack - runs beside the MMAs on sixteen warps, 400 cycles a chunk, and is the longer part
// of 1 x 1 layers alone (512 x 64 -> 64 on 25 x 5: 7.4 us, tensor pipe 2 %).  Half of its shared-memory wavefronts are bank
// conflicts: lanes of different border classes read rows of the same banks.  The 4-way byte dot products on CUDA cores that
// ran such layers before took 258 us.
#include <cuda.h>

#include <cstring>
#include <string>
#include <unordered_map>

#include "common.cuh"
#include "sm100.cuh"

namespace small {

namespace {

using namespace sm100;

constexpr int kEpi = 4;                    // epilogue groups of four warps
constexpr int kThreads = 128 + 128 * kEpi;
constexpr int kMaxA = 8, kMaxB = 16;       // strip stages, streamed filter boxes
constexpr int kMaxSlots = 8;
constexpr int kTmemCols = 512;
constexpr int kOnesRows = 16;              // rows behind the filters of a box: one of ones, the rest zero (N is a multiple of 16)
constexpr int kMaxTaps = 256;

struct I8Args {
    uint8_t *out; const uint8_t *w; const int *bias; const int *w_sums;     // w_sums: [K][T] sums of weight bytes over the channels
    int *status;
    int N, C, K, KB, CB, T, FH, FW, S, pt, pl, pb, pr, H, W;      // the layer
    int OH, OW;                              // output plane as the tiles see it (one row for a pointwise layer)
    int Wq, Hq, nn, rows, tw, tiles_w, bands, m_tiles, n_tiles, Kt, cols, slots, slot_cols, epi, n_phase, phase_bits, dh0, dw0;
    int FHv, FWv, ptv, plv;                  // the stride-1 view's window and pads
    int strip_px, tail_px, loads, load_rows; // strips may take several boxes (very tall windows)
    uint32_t a_stage, a_box, b_box;          // bytes: strip stage, one input box, one filter box with its extra rows
    int a_stages, b_stages, resident;
    int row_classes, col_classes;            // border classes tabulated (0: none, border pixels sum their taps themselves)
    int zx, zw, zo, mult, shift, lo;
    uint32_t wait_iters;
    // taps sorted by phase plane: strip offset in 16-byte units, original tap; phase p holds entries phase_at[p] .. [p + 1] - 1
    int phase_at[5];
    uint16_t tap_off[kMaxTaps];
    uint8_t tap_id[kMaxTaps];
};

// Shared-memory matrix descriptor, K-major, 32-byte swizzle: rows 32 bytes apart, groups of 8 rows 256 bytes apart.
constexpr uint32_t kDescHi32 = (256u >> 4) | (1u << 14) | (6u << 29);

__device__ __forceinline__ void mma_i8(uint32_t d, uint32_t a_lo, uint32_t b_lo, uint32_t idesc, uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t.reg .b64 da, db;\n\t"
        "setp.ne.b32 p, %5, 0;\n\t"
        "mov.b64 da, {%1, %3};\n\t"
        "mov.b64 db, {%2, %3};\n\t"
        "tcgen05.mma.cta_group::1.kind::i8 [%0], da, db, %4, p;\n\t}"
        ::"r"(d), "r"(a_lo), "r"(b_lo), "r"(kDescHi32), "r"(idesc), "r"(accumulate) : "memory");
}
__device__ __forceinline__ int tmem_ld1(uint32_t taddr) {
    uint32_t r;
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x1.b32 {%0}, [%1];" : "=r"(r) : "r"(taddr) : "memory");
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
    return (int)r;
}

struct I8Tile { int n0, oh0, ow0, px; };

__device__ __forceinline__ I8Tile decode(const I8Args &a, int m) {
    I8Tile t;
    if (a.nn > 1) { t.n0 = m * a.nn; t.oh0 = 0; t.ow0 = 0; t.px = min(a.nn, a.N - t.n0) * a.Hq * a.Wq; return t; }
    int r = m;
    t.ow0 = 0;
    if (a.tiles_w > 1) { const int wt = r % a.tiles_w; r /= a.tiles_w; t.ow0 = wt * a.tw; }
    t.n0 = r / a.bands;
    t.oh0 = (r - t.n0 * a.bands) * a.rows;
    t.px = min(a.rows, a.OH - t.oh0) * a.Wq;
    return t;
}

// CH: 128-pixel chunks per tile
template <int CH>
__global__ void __launch_bounds__(kThreads, 1)
conv_i8_kernel(const __grid_constant__ CUtensorMap map_a, const __grid_constant__ I8Args a) {
    extern __shared__ uint8_t smem_raw[];
    __shared__ __align__(8) unsigned long long bars[2 * kMaxA + 2 * kMaxB + 2 * kMaxSlots];
    __shared__ uint32_t tmem_addr;
    __shared__ volatile int abort_flag;
    const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    uint8_t *bp = smem_raw + (base - smem_u32(smem_raw));
    const uint32_t b_base = base + a.a_stages * a.a_stage;
    uint8_t *tab = bp + (size_t)a.a_stages * a.a_stage + (size_t)a.b_stages * a.b_box;
    long long *addend = reinterpret_cast<long long *>(tab);                       // [Kt] bias * mult + half
    int *w_tab = reinterpret_cast<int *>(tab + (size_t)a.Kt * 8);                 // [Kt][T]
    int *cst = reinterpret_cast<int *>(tab + (size_t)a.Kt * 8 + (((size_t)a.Kt * a.T * 4 + 15) & ~(size_t)15));   // [class][Kt]
    const uint32_t bar0 = smem_u32(bars);
    const uint32_t a_full = bar0, a_empty = a_full + 8 * kMaxA, b_full = a_empty + 8 * kMaxA, b_empty = b_full + 8 * kMaxB;
    const uint32_t slot_full = b_empty + 8 * kMaxB, slot_free = slot_full + 8 * kMaxSlots;
    const int warp = warp_index(), lane = threadIdx.x & 31;
    const int nt = a.n_tiles > 1 ? (int)(blockIdx.x % a.n_tiles) : 0;             // this block's filter tile
    const int m_first = a.n_tiles > 1 ? (int)(blockIdx.x / a.n_tiles) : (int)blockIdx.x, m_step = gridDim.x / a.n_tiles;
    const int k_tile = nt * a.Kt;

    if (threadIdx.x == 0) {
        for (int s = 0; s < a.a_stages; ++s) { mbar_init(a_full + 8 * s, 1); mbar_init(a_empty + 8 * s, 1); }
        for (int s = 0; s < (a.resident ? 1 : a.b_stages); ++s) { mbar_init(b_full + 8 * s, 1); mbar_init(b_empty + 8 * s, 1); }
        // every chunk of a tile belongs to one epilogue group (four warps)
        for (int s = 0; s < a.slots; ++s) { mbar_init(slot_full + 8 * s, 1); mbar_init(slot_free + 8 * s, 4 * CH); }
        abort_flag = 0;
        mbar_fence_init();
    }
    if (warp == 1) tmem_alloc(smem_u32(&tmem_addr), kTmemCols);
    // extra rows of every filter box (TMA never writes them): a row of ones, then zeros
    for (int i = threadIdx.x; i < a.b_stages * kOnesRows * 2; i += kThreads) {
        const int box = i / (kOnesRows * 2), r = i - box * kOnesRows * 2;
        const uint32_t v = r < 2 ? 0x01010101u : 0u;
        reinterpret_cast<uint4 *>(bp + (b_base - base) + (size_t)box * a.b_box + (size_t)a.Kt * 32)[r] = make_uint4(v, v, v, v);
    }
    // zero tail behind each strip: the padding the last row (or image) wraps into
    if (a.tail_px)
        for (int i = warp; i < a.a_stages * a.tail_px; i += kThreads / 32)
            if (lane < 2) reinterpret_cast<uint4 *>(bp + (size_t)(i % a.a_stages) * a.a_stage + (size_t)(a.strip_px + i / a.a_stages) * 32)[lane] = make_uint4(0u, 0u, 0u, 0u);
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_addr;
    grid_dep_sync();
    grid_dep_trigger();

    const int blocks = a.n_phase * a.CB;
    uint32_t armed = 0, armed_par = 0, drain = 0;
    if (warp == 0) {
        // ---- input strips: one per (tile, phase plane, channel block)
        drain = a_full;
        bool alive = true, wrapped = false;
        uint32_t s = 0, ph = 0;
        for (int m = m_first; m < a.m_tiles && alive; m += m_step) {
            const I8Tile t = decode(a, m);
            for (int p = 0; p < a.n_phase && alive; ++p) {
                const int x = a.S * (t.ow0 - a.plv) + ((a.phase_bits >> (2 * p + 1)) & 1), y = a.S * (t.oh0 - a.ptv) + ((a.phase_bits >> (2 * p)) & 1);
                for (int cb = 0; cb < a.CB; ++cb) {
                    if (wrapped) alive = mbar_wait_uniform<4>(a_empty + 8 * s, ph ^ 1u, &abort_flag, a.status, a.wait_iters);
                    if (!alive) break;
                    if (elect_one()) {
                        mbar_expect_tx(a_full + 8 * s, a.a_box * a.loads);
                        for (int l = 0; l < a.loads; ++l)
                            tma_load_5d(base + s * a.a_stage + l * a.a_box, &map_a, a_full + 8 * s, 0, x, y + a.S * l * a.load_rows, cb, t.n0);
                    }
                    armed |= 1u << s;
                    armed_par = (armed_par & ~(1u << s)) | (ph << s);
                    if (++s == (uint32_t)a.a_stages) { s = 0; ph ^= 1u; wrapped = true; }
                }
            }
        }
    } else if (warp == 2) {
        // ---- filter boxes: one per (phase plane, channel block, tap)
        drain = b_full;
        // (a last filter tile with fewer filters leaves rows of its boxes as they are: columns nobody reads)
        const uint32_t bytes = (uint32_t)min(a.Kt, a.KB * 32 - k_tile) * 32u;
        const uint8_t *w0 = a.w + (size_t)k_tile * 32;
        if (a.resident) {
            if (elect_one()) {
                mbar_expect_tx(b_full, bytes * (uint32_t)(a.CB * a.T));
                uint32_t dst = b_base;
                for (int p = 0; p < a.n_phase; ++p)
                    for (int cb = 0; cb < a.CB; ++cb)
                        for (int i = a.phase_at[p]; i < a.phase_at[p + 1]; ++i, dst += a.b_box) bulk_load(dst, w0 + (size_t)(cb * a.T + a.tap_id[i]) * a.KB * 1024, bytes, b_full);
            }
            armed = 1u;
        } else {
            bool alive = true, wrapped = false;
            uint32_t s = 0, ph = 0;
            for (int m = m_first; m < a.m_tiles && alive; m += m_step)
                for (int p = 0; p < a.n_phase && alive; ++p)
                    for (int cb = 0; cb < a.CB && alive; ++cb)
                        for (int i = a.phase_at[p]; i < a.phase_at[p + 1]; ++i) {
                            if (wrapped) alive = mbar_wait_uniform<4>(b_empty + 8 * s, ph ^ 1u, &abort_flag, a.status, a.wait_iters);
                            if (!alive) break;
                            if (elect_one()) {
                                mbar_expect_tx(b_full + 8 * s, bytes);
                                bulk_load(b_base + s * a.b_box, w0 + (size_t)(cb * a.T + a.tap_id[i]) * a.KB * 1024, bytes, b_full + 8 * s);
                            }
                            armed |= 1u << s;
                            armed_par = (armed_par & ~(1u << s)) | (ph << s);
                            if (++s == (uint32_t)a.b_stages) { s = 0; ph ^= 1u; wrapped = true; }
                        }
        }
    } else if (warp == 1) {
        // ---- MMA issue
        // instruction descriptor: S32 accumulator, U8 A and B, both K-major, M = 128, N = filters + extra rows
        const uint32_t idesc = (2u << 4) | ((uint32_t)((a.Kt + kOnesRows) >> 3) << 17) | ((128u >> 4) << 24);
        const uint32_t elected = elect_one();
        bool alive = true;
        uint32_t sa = 0, pa = 0, sb = 0, pb = 0, slot = 0, slot_par = 1;
        const uint32_t b_step = a.b_box >> 4;
        if (a.resident) alive = mbar_wait_uniform(b_full, 0, &abort_flag, a.status, a.wait_iters);
        for (int m = m_first; m < a.m_tiles && alive; m += m_step) {
            alive = mbar_wait_uniform(slot_free + 8 * slot, slot_par, &abort_flag, a.status, a.wait_iters);   // passes at once in the first round
            if (!alive) break;
            tc_fence_after();
            const uint32_t acc0 = tmem + slot * (uint32_t)a.slot_cols;
            uint32_t w_lo = smem_desc_lo(b_base), first = 0;
            int p = 0, cb = 0;
            for (int blk = 0; blk < blocks && alive; ++blk) {
                alive = mbar_wait_uniform(a_full + 8 * sa, pa, &abort_flag, a.status, a.wait_iters);
                if (!alive) break;
                tc_fence_after();
                const uint32_t x0 = smem_desc_lo(base + sa * a.a_stage);
                const int i1 = a.phase_at[p + 1];
                // The loop over the taps holds nothing but address steps and MMAs: with the code of the streamed filters' wait
                // inside it, jumped over, each iteration took 390 cycles instead of 80 (instruction fetches).
                if (a.resident) {
                    for (int i = a.phase_at[p]; i < i1; ++i) {
                        const uint32_t xo = x0 + a.tap_off[i];
                        if (elected) {
#pragma unroll
                            for (int c = 0; c < CH; ++c) mma_i8(acc0 + (uint32_t)(c * a.cols), xo + c * 256u, w_lo, idesc, first);
                        }
                        first = 1u;
                        w_lo += b_step;
                    }
                } else {
                    for (int i = a.phase_at[p]; i < i1; ++i) {
                        alive = mbar_wait_uniform(b_full + 8 * sb, pb, &abort_flag, a.status, a.wait_iters);
                        if (!alive) break;
                        const uint32_t xo = x0 + a.tap_off[i], ws = smem_desc_lo(b_base + sb * a.b_box);
                        if (elected) {
#pragma unroll
                            for (int c = 0; c < CH; ++c) mma_i8(acc0 + (uint32_t)(c * a.cols), xo + c * 256u, ws, idesc, first);
                            mma_commit(b_empty + 8 * sb);
                        }
                        first = 1u;
                        if (++sb == (uint32_t)a.b_stages) { sb = 0; pb ^= 1u; }
                    }
                }
                if (alive && elected) mma_commit(a_empty + 8 * sa);
                if (++sa == (uint32_t)a.a_stages) { sa = 0; pa ^= 1u; }
                if (++cb == a.CB) { cb = 0; ++p; }
            }
            if (alive && elected) mma_commit(slot_full + 8 * slot);
            if (++slot == (uint32_t)a.slots) { slot = 0; slot_par ^= 1u; }
        }
    } else if (warp >= 4) {
        // ---- tables of this block's filter tile
        constexpr int kEt = 128 * kEpi;
        const int et = threadIdx.x - 128;
        const int n_real = min(a.Kt, a.K - k_tile);
        const int cr = a.pb + 1, cc = a.pr + 1;
        const int classes = a.row_classes * a.col_classes;
        const bool zo_in = a.shift >= 32 && a.shift <= 43;       // see the requantisation below
        for (int k = et; k < a.Kt; k += kEt)
            addend[k] = (a.bias && k < n_real ? (long long)a.bias[k_tile + k] * a.mult : 0ll) + (1ll << (a.shift - 1)) + (zo_in ? (long long)a.zo << a.shift : 0ll);
        // the terms of the identity above that depend on the filter and the taps rows [x0, x1) x columns [y0, y1)
        const uint32_t zz = (uint32_t)(a.C * a.zx * a.zw);
        auto taps_const = [&](int k, int x0, int x1, int y0, int y1) {
            uint32_t s = 0;
            for (int x = x0; x < x1; ++x)
                for (int y = y0; y < y1; ++y) s += (uint32_t)w_tab[k * a.T + x * a.FW + y];
            return (int)((uint32_t)((x1 - x0) * (y1 - y0)) * zz - (uint32_t)a.zx * s);
        };
        if (classes && a.FH <= 3) {
            // windows up to 3 x 3: a thread holds its filter's tap sums in registers and takes every so many classes
            const int groups = kEt / a.Kt, first = et / a.Kt, k = et - first * a.Kt;
            uint32_t ws[3][3];
#pragma unroll
            for (int x = 0; x < 3; ++x)
#pragma unroll
                for (int y = 0; y < 3; ++y)
                    ws[x][y] = (k < n_real && x < a.FH && y < a.FW) ? (uint32_t)a.w_sums[(size_t)(k_tile + k) * a.T + x * a.FW + y] : 0u;
            int cl = 0, next = first;
            for (int xt = 0; xt <= a.pt; ++xt)
                for (int xb = 0; xb <= a.pb; ++xb) {
                    const int rows_in = max(0, a.FH - xb - xt);
                    for (int yl = 0; yl <= a.pl; ++yl)
                        for (int yr = 0; yr <= a.pr; ++yr, ++cl) {
                            if (cl != next) continue;
                            next += groups;
                            uint32_t s = 0;
#pragma unroll
                            for (int x = 0; x < 3; ++x)
#pragma unroll
                                for (int y = 0; y < 3; ++y) s += (x >= xt && x < a.FH - xb && y >= yl && y < a.FW - yr) ? ws[x][y] : 0u;
                            cst[cl * a.Kt + k] = (int)((uint32_t)(rows_in * max(0, a.FW - yr - yl)) * zz - (uint32_t)a.zx * s);
                        }
                }
        } else {
            for (int i = et; i < a.Kt * a.T; i += kEt) w_tab[i] = i < n_real * a.T ? a.w_sums[(size_t)k_tile * a.T + i] : 0;
            asm volatile("bar.sync 1, 512;" ::: "memory");
            for (int i = et; i < (classes ? classes : 1) * a.Kt; i += kEt) {
                const int cl = i / a.Kt, k = i - cl * a.Kt;
                const int rc = classes ? cl / a.col_classes : 0, ccl = classes ? cl - rc * a.col_classes : 0;
                const int x0 = rc / cr, x1 = a.FH - rc % cr, y0 = ccl / cc, y1 = a.FW - ccl % cc;
                cst[i] = (x0 < x1 && y0 < y1) ? taps_const(k, x0, x1, y0, y1) : 0;
            }
        }
        asm volatile("bar.sync 1, 512;" ::: "memory");

        const int quarter = warp & 3, group = (warp - 4) >> 2;
        bool alive = true;
        uint32_t slot = 0, slot_par = 0, turn = 0;
        const int pv = a.Hq * a.Wq;
        for (int m = m_first; m < a.m_tiles && alive; m += m_step) {
            const uint32_t s = slot, par = slot_par;
            if (++slot == (uint32_t)a.slots) { slot = 0; slot_par ^= 1u; }
            // The groups take the chunks in turn.  (A group waits for a slot's fill by its parity, which says nothing unless
            // the fill before that one is known to be over: so no more groups than chunks in all slots.)
            if (group >= a.epi) break;
            const int c_mine = (group - (int)turn) & (a.epi - 1);
            turn = (turn + CH) & (uint32_t)(a.epi - 1);
            if (c_mine >= CH) continue;
            const I8Tile t = decode(a, m);
            alive = mbar_wait_warp<8>(slot_full + 8 * s, par, &abort_flag, a.status, a.wait_iters);
            if (!alive) break;
            tc_fence_after();
            if (c_mine * 128 < t.px) {
                const int c = c_mine;
                const uint32_t taddr = tmem + s * (uint32_t)a.slot_cols + (uint32_t)(c * a.cols) + ((uint32_t)(quarter * 32) << 16);
                int q = c * 128 + quarter * 32 + lane, img = 0;
                const bool in_tile = q < t.px;
                if (a.nn > 1) { img = q / pv; q -= img * pv; }
                const int r = q / a.Wq, oh = t.oh0 + r, ow = t.ow0 + q - r * a.Wq;
                const bool ok = in_tile && oh < a.OH && ow < min(a.OW, t.ow0 + a.tw);
                const int n = t.n0 + img;
                // window rows and columns outside the plane (none for a pointwise layer, whose plane the tiles see as one row)
                const int ih = oh * a.S - a.pt, iw = ow * a.S - a.pl;
                int x0 = 0, xm = 0, y0 = 0, ym = 0;
                if (ok && a.pt + a.pb + a.pl + a.pr > 0) {
                    x0 = max(0, -ih); xm = max(0, ih + a.FH - a.H);
                    y0 = max(0, -iw); ym = max(0, iw + a.FW - a.W);
                }
                const int cl = classes ? (x0 * cr + xm) * a.col_classes + y0 * cc + ym : 0;
                const int zsx = a.zw * tmem_ld1(taddr + a.Kt);
                for (int j = 0; j * 32 < a.Kt; ++j) {
                    float vf[32];
                    tmem_ld32(taddr + j * 32, vf);
                    const int kb = (k_tile >> 5) + j;
                    if (!ok || kb >= a.KB) continue;
                    int sum[32];
                    const int4 *c4 = reinterpret_cast<const int4 *>(cst + cl * a.Kt + j * 32);
#pragma unroll
                    for (int i = 0; i < 8; ++i) {
                        const int4 cv = c4[i];
                        sum[4 * i] = cv.x + __float_as_int(vf[4 * i]) - zsx; sum[4 * i + 1] = cv.y + __float_as_int(vf[4 * i + 1]) - zsx;
                        sum[4 * i + 2] = cv.z + __float_as_int(vf[4 * i + 2]) - zsx; sum[4 * i + 3] = cv.w + __float_as_int(vf[4 * i + 3]) - zsx;
                    }
                    if (!classes && (x0 | xm | y0 | ym)) {       // too many border classes for a table: this pixel's own taps
#pragma unroll 1
                        for (int e = 0; e < 32; ++e) {
                            const int d = taps_const(j * 32 + e, x0, a.FH - xm, y0, a.FW - ym) - cst[j * 32 + e];
#pragma unroll
                            for (int i = 0; i < 32; ++i) sum[i] += i == e ? d : 0;
                        }
                    }
                    const longlong2 *ad = reinterpret_cast<const longlong2 *>(addend + j * 32);
                    // Requantisation: the addend holds bias * mult, the rounding half and, for 32 <= shift <= 43, the output's
                    // zero point << shift: |acc + bias| * mult + all of it stays below 2^63 there (|acc| <= 33000 * 255^2).
                    uint32_t word[8];
                    if (zo_in) {
                        const int sh = a.shift - 32;
#pragma unroll
                        for (int i = 0; i < 16; ++i) {
                            const longlong2 av = ad[i];
                            const int v0 = max((int)(((long long)sum[2 * i] * (long long)a.mult + av.x) >> 32) >> sh, a.lo);
                            const int v1 = max((int)(((long long)sum[2 * i + 1] * (long long)a.mult + av.y) >> 32) >> sh, a.lo);
                            uint32_t two;                            // both saturated to bytes
                            asm("cvt.pack.sat.u8.s32.b32 %0, %1, %2, %3;" : "=r"(two) : "r"(v1), "r"(v0), "r"(0u));
                            word[i >> 1] = (i & 1) ? __byte_perm(word[i >> 1], two, 0x5410) : two;
                        }
                    } else {
#pragma unroll
                        for (int i = 0; i < 8; ++i) {
                            uint32_t w4 = 0;
#pragma unroll
                            for (int e = 0; e < 4; ++e) {
                                const long long r = (((long long)sum[4 * i + e] * (long long)a.mult + addend[j * 32 + 4 * i + e]) >> a.shift) + a.zo;
                                w4 |= (uint32_t)(r < a.lo ? a.lo : r > 255 ? 255 : (int)r) << (8 * e);
                            }
                            word[i] = w4;
                        }
                    }
                    const int left = a.K - kb * 32;                                // pad lanes stay 0
                    if (left < 32) {
#pragma unroll
                        for (int i = 0; i < 8; ++i) {
                            const int n_ok = left - 4 * i;
                            word[i] = n_ok >= 4 ? word[i] : n_ok <= 0 ? 0u : word[i] & ((1u << (8 * n_ok)) - 1u);
                        }
                    }
                    uint8_t *dst = a.out + (((size_t)n * a.KB + kb) * a.OH * a.OW + (size_t)oh * a.OW + ow) * 32;
                    reinterpret_cast<uint4 *>(dst)[0] = make_uint4(word[0], word[1], word[2], word[3]);
                    reinterpret_cast<uint4 *>(dst)[1] = make_uint4(word[4], word[5], word[6], word[7]);
                }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(slot_free + 8 * s);
        }
        tc_fence_before();
    }
    __syncthreads();
    if (abort_flag && armed && lane == 0) {   // a role gave up: let the copies in flight land before the block exits
        for (int st = 0; st < 32; ++st)
            if (armed >> st & 1u)
                for (uint32_t it = 0; it < a.wait_iters && !mbar_try_wait(drain + 8 * st, armed_par >> st & 1u); ++it) __nanosleep(200);
    }
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem, kTmemCols);
    }
}

// ---------------------------------------------------------------------------------------------- host side
struct I8Plan { I8Args a; int ch; unsigned grid; size_t smem; bool ok; };

int floor_half(int v) { return v >= 0 ? v / 2 : -((1 - v) / 2); }

// The cheapest tiling over the chunks per tile (1, 2 or 4) and the filters per tile (32 to 128).  Where the filter tiles share
// the SMs, a block of each walks its part of the pixel tiles; more filter tiles than SMs (above 18,944 filters on 148 SMs, any
// tiling) take one block each, which walks all pixel tiles, and the blocks follow one another over the SMs.
I8Plan plan_i8(const Geom &g, size_t max_smem, int sms) {
    I8Plan best{};
    best.ok = false;
    if ((g.FW != 1 && g.FW != 3) || (g.S != 1 && g.S != 2) || g.FH * g.FW > kMaxTaps) return best;
    I8Args b{};
    b.N = g.N; b.C = g.C; b.K = g.K; b.KB = g.KB; b.CB = g.CB; b.T = g.FH * g.FW; b.FH = g.FH; b.FW = g.FW; b.S = g.S;
    b.pt = g.pt; b.pl = g.pl; b.pb = g.pb; b.pr = g.pr; b.H = g.H; b.W = g.W; b.OH = g.OH; b.OW = g.OW;
    // the stride-1 view (see conv_tc.cu)
    int Hv = g.H, Wv = g.W, pbv = g.pb, prv = g.pr;
    b.FHv = g.FH; b.FWv = g.FW; b.ptv = g.pt; b.plv = g.pl; b.n_phase = 1; b.phase_bits = 0;
    if (g.S == 2) {
        b.dh0 = floor_half(-g.pt); b.dw0 = floor_half(-g.pl);
        b.FHv = floor_half(g.FH - 1 - g.pt) - b.dh0 + 1; b.FWv = floor_half(g.FW - 1 - g.pl) - b.dw0 + 1;
        b.ptv = -b.dh0; b.plv = -b.dw0; pbv = prv = 0;
        bool hh[2] = {false, false}, hw[2] = {false, false};
        for (int x = 0; x < g.FH; ++x) hh[(x - g.pt) & 1] = true;
        for (int y = 0; y < g.FW; ++y) hw[(y - g.pl) & 1] = true;
        b.n_phase = 0;
        for (int ph = 0; ph < 2; ++ph)
            for (int pw = 0; pw < 2; ++pw)
                if (hh[ph] && hw[pw]) b.phase_bits |= (ph | (pw << 1)) << (2 * b.n_phase++);
        Hv = g.OH + b.FHv - 1 - b.ptv; Wv = g.OW + b.FWv - 1 - b.plv;
    } else if (b.T == 1 && !(g.pt | g.pb | g.pl | g.pr)) {      // pointwise: the plane is one row of pixels
        b.OW = Wv = g.H * g.W; b.OH = Hv = 1;
    }
    const int maxw = b.plv > prv ? b.plv : prv, minw = b.plv < prv ? b.plv : prv;
    const int maxh = b.ptv > pbv ? b.ptv : pbv, minh = b.ptv < pbv ? b.ptv : pbv;
    const int lim = 256 / g.S;                                   // pixels a box spans in one dimension
    double best_cost = 0.0;
    for (int many = 0; many < 2 && !best.ok; ++many)         // first tilings of no more filter tiles than SMs, else any
    for (int ch = 4; ch >= 1; ch >>= 1) {
        I8Args a = b;
        const int px = ch * 128;
        const long long pv = (long long)(Hv + maxh) * (Wv + maxw);
        if (pv * 2 <= px && Hv + maxh <= lim && Wv + maxw <= lim) {
            a.Wq = Wv + maxw; a.Hq = Hv + maxh;                   // whole images, the padding between neighbours shared
            a.nn = (int)(px / pv);
            if (a.nn > g.N) a.nn = g.N;
            if (a.nn > 256) a.nn = 256;
        }
        if (a.nn <= 1) a.nn = 1;
        if (a.nn > 1) {
            a.rows = a.OH; a.tw = a.OW; a.tiles_w = 1; a.bands = 1; a.m_tiles = ceil_div(g.N, a.nn);
            a.loads = 1; a.load_rows = a.Hq;
            a.strip_px = a.nn * a.Hq * a.Wq;
            a.tail_px = minh * a.Wq + minw;
        } else {
            // bands of whole rows of one image; wide planes are cut into column tiles
            a.tiles_w = ceil_div(a.OW, px);
            for (;; ++a.tiles_w) {
                a.tw = ceil_div(a.OW, a.tiles_w);
                a.Wq = a.tiles_w == 1 ? Wv + maxw : a.tw + a.FWv - 1;
                a.rows = a.Wq > px ? 0 : px / a.Wq;
                if (a.rows > a.OH) a.rows = a.OH;
                if (a.FHv <= lim && a.rows + a.FHv - 1 > lim) a.rows = lim - a.FHv + 1;
                if (a.rows >= 1 && a.Wq <= lim && (size_t)(a.rows + a.FHv - 1) * a.Wq * 32 <= 40 * 1024) break;
                if (a.tw == 1) { a.rows = 0; break; }
            }
            if (a.rows < 1) continue;
            a.tiles_w = ceil_div(a.OW, a.tw);
            a.bands = ceil_div(a.OH, a.rows);
            a.rows = ceil_div(a.OH, a.bands);
            const long long m = (long long)g.N * a.bands * a.tiles_w;
            if (m > 0x3fffffff) continue;
            a.m_tiles = (int)m;
            const int Rs = a.rows + a.FHv - 1;
            a.Hq = Rs;
            a.loads = 1; a.load_rows = Rs;
            if (Rs > lim) { a.load_rows = lim / 2; a.loads = ceil_div(Rs, a.load_rows); }    // (boxes of a multiple of 8 rows: swizzle phase)
            a.strip_px = a.loads * a.load_rows * a.Wq;
            a.tail_px = a.tiles_w == 1 ? minw : 0;
        }
        const int reach = px + (a.FHv - 1) * a.Wq + a.FWv - 1;    // furthest pixel an MMA reads
        const int stage_px = a.strip_px + a.tail_px > reach ? a.strip_px + a.tail_px : reach;
        a.a_stage = (uint32_t)(((size_t)stage_px * 32 + 1023) & ~(size_t)1023);
        a.a_box = (uint32_t)((a.loads > 1 ? a.load_rows * a.Wq : a.strip_px) * 32);
        const long long classes = (long long)(g.pt + 1) * (g.pb + 1) * (g.pl + 1) * (g.pr + 1);
        for (int kt = 32; kt <= 128 && kt < g.KB * 32 + 32; kt += 32) {
            a.Kt = kt;
            a.cols = kt + 32;
            // accumulator slots: as many as tensor memory holds, at least two
            a.slot_cols = ch * a.cols;
            a.slots = kTmemCols / a.slot_cols;
            if (a.slots < 2) continue;
            if (a.slots > kMaxSlots) a.slots = kMaxSlots;
            a.epi = a.slots * ch >= kEpi ? kEpi : 2;
            a.n_tiles = ceil_div(g.KB * 32, kt);
            if ((a.n_tiles > sms) != (many == 1)) continue;
            a.b_box = (uint32_t)(kt + kOnesRows) * 32u;
            const bool table = classes * kt * 4 <= 32 * 1024;
            a.row_classes = table ? (g.pt + 1) * (g.pb + 1) : 0; a.col_classes = table ? (g.pl + 1) * (g.pr + 1) : 0;
            const size_t fixed = 1024 + (size_t)kt * 8 + (((size_t)kt * a.T * 4 + 15) & ~(size_t)15) + (size_t)(table ? classes : 1) * kt * 4;
            const size_t all_b = (size_t)a.CB * a.T * a.b_box;
            const size_t room = max_smem - 2 * 1024;             // static shared memory: barriers
            a.resident = fixed + all_b + 3 * (size_t)a.a_stage <= room;
            a.b_stages = a.resident ? a.CB * a.T : 0;
            if (!a.resident) {
                a.b_stages = kMaxB;
                while (a.b_stages > 2 && fixed + (size_t)a.b_stages * a.b_box + 3 * (size_t)a.a_stage > room) --a.b_stages;
            }
            const size_t used = fixed + (size_t)a.b_stages * a.b_box;
            if (used + 2 * (size_t)a.a_stage > room) continue;
            a.a_stages = (int)((room - used) / a.a_stage);
            if (a.a_stages > kMaxA) a.a_stages = kMaxA;
            // cycles of the busiest block: MMAs (128 x N x 32: 32 + N / 4 cycles of operand reads, some more to issue)
            // beside the requantisation (about 350 cycles per 128 pixels and 32 filters for one group of four warps)
            const int per = many ? 1 : sms / a.n_tiles;
            const double tiles = (double)ceil_div(a.m_tiles, per < a.m_tiles ? per : a.m_tiles) * ceil_div(a.n_tiles, sms);
            const double mma = (double)ch * a.CB * a.T * (48.0 + (kt + kOnesRows) / 4.0);
            const double epi = (double)ch * (kt / 32) * (a.epi == kEpi ? 200.0 : 300.0);
            const double load = ((double)a.CB * a.n_phase * a.strip_px * 32 + (a.resident ? 0.0 : (double)all_b)) / 40.0;
            double tile = mma > epi ? mma : epi;
            if (load > tile) tile = load;
            const double cost = tiles * (tile + 250.0) + (mma < epi ? mma : epi) + (a.resident ? (double)all_b / 40.0 : 0.0);
            if (!best.ok || cost < best_cost) {
                best.ok = true; best_cost = cost;
                best.a = a; best.ch = ch;
                const int blocks_m = a.m_tiles < per ? a.m_tiles : per;
                best.grid = (unsigned)(blocks_m * a.n_tiles);
                best.smem = used + (size_t)a.a_stages * a.a_stage;
            }
        }
    }
    return best;
}

struct I8Launch { CUtensorMap map_a; I8Args a; int ch; unsigned grid; size_t smem; };
typedef std::unordered_map<std::string, I8Launch> I8Cache;

int start(small_ctx *ctx, const I8Launch &L, cudaStream_t st) {
    auto kern = L.ch == 4 ? conv_i8_kernel<4> : L.ch == 2 ? conv_i8_kernel<2> : conv_i8_kernel<1>;
    launch_kernel(ctx, kern, dim3(L.grid), dim3(kThreads), L.smem, st, L.map_a, L.a);
    return check_launch(ctx);
}

}  // namespace

void free_i8_cache(small_ctx *ctx) {
    delete static_cast<I8Cache *>(ctx->i8_cache);
    ctx->i8_cache = nullptr;
}

int launch_q_conv(small_ctx *ctx, const uint8_t *in, const uint8_t *w, const int *w_sums, const int *bias, uint8_t *out, const Geom &g,
                  bool relu, int zx, int zw, int zo, int mult, int shift, cudaStream_t st) {
    // a launch seen before (same shape, parameters and tensors): everything is ready
    const int ints[] = {g.N, g.C, g.K, g.H, g.W, g.FH, g.FW, g.S, g.pt, g.pb, g.pl, g.pr, relu ? 1 : 0, zx, zw, zo, mult, shift, (int)ctx->wait_iters};
    const void *ptrs[] = {in, w, bias, out};
    std::string key(reinterpret_cast<const char *>(ints), sizeof(ints));
    key.append(reinterpret_cast<const char *>(ptrs), sizeof(ptrs));
    if (!ctx->i8_cache) ctx->i8_cache = new I8Cache();
    I8Cache &cache = *static_cast<I8Cache *>(ctx->i8_cache);
    auto it = cache.find(key);
    if (it != cache.end()) return start(ctx, it->second, st);
    I8Plan p = plan_i8(g, ctx->max_smem_optin, ctx->sm_count);
    if (!p.ok) return SMALL_ERR_UNSUPPORTED;
    I8Launch L;
    L.a = p.a; L.ch = p.ch; L.grid = p.grid; L.smem = p.smem;
    I8Args &a = L.a;
    a.out = out; a.w = w; a.bias = bias; a.w_sums = w_sums; a.status = ctx->dev_status; a.wait_iters = ctx->wait_iters;
    a.zx = zx; a.zw = zw; a.zo = zo; a.mult = mult; a.shift = shift; a.lo = relu ? zo : 0;
    EncodeTiledFn encode = reinterpret_cast<EncodeTiledFn>(ctx->encode_tiled);
    {   // activations [N][CB][H][W][32 bytes]
        const bool flat = a.OH == 1 && a.T == 1 && g.S == 1 && a.OW == g.H * g.W;
        const cuuint64_t W = flat ? (cuuint64_t)g.H * g.W : g.W, H = flat ? 1 : g.H;
        const cuuint32_t es = (cuuint32_t)g.S;
        cuuint64_t dims[5] = {32, W, H, (cuuint64_t)g.CB, (cuuint64_t)g.N};
        cuuint64_t strides[4] = {32, W * 32, W * H * 32, (cuuint64_t)g.CB * W * H * 32};
        cuuint32_t box[5] = {32, (cuuint32_t)a.Wq * es, (cuuint32_t)a.load_rows * es, 1, (cuuint32_t)a.nn};
        cuuint32_t estr[5] = {1, es, es, 1, 1};
        CUresult r = encode(&L.map_a, CU_TENSOR_MAP_DATA_TYPE_UINT8, 5, const_cast<uint8_t *>(in), dims, strides, box, estr,
                            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_32B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
        if (r != CUDA_SUCCESS) { ctx->last_cuda = (int)r; return SMALL_ERR_CUDA; }
    }
    // tap (x, y) reads row oh + floor((x - pt) / S) of phase plane ((x - pt) mod S, (y - pl) mod S)
    for (int p = 0, n = 0; p < a.n_phase; ++p) {
        for (int x = 0; x < g.FH; ++x)
            for (int y = 0; y < g.FW; ++y) {
                int px = x * a.Wq + y, bits = 0;
                if (g.S == 2) {
                    bits = ((x - g.pt) & 1) | (((y - g.pl) & 1) << 1);
                    px = (floor_half(x - g.pt) - a.dh0) * a.Wq + floor_half(y - g.pl) - a.dw0;
                }
                if (bits != ((a.phase_bits >> (2 * p)) & 3)) continue;
                a.tap_off[n] = (uint16_t)(px * 2); a.tap_id[n] = (uint8_t)(x * g.FW + y);
                ++n;
            }
        a.phase_at[p + 1] = n;
    }
    auto kern = L.ch == 4 ? conv_i8_kernel<4> : L.ch == 2 ? conv_i8_kernel<2> : conv_i8_kernel<1>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)ctx->max_smem_optin - 2 * 1024);
    if (e != cudaSuccess) { ctx->last_cuda = (int)e; return SMALL_ERR_CUDA; }
    if (cache.size() >= 4096) cache.clear();
    cache[key] = L;
    return start(ctx, L, st);
}

}  // namespace small
