// Single channel reduction with weights (paper Section 3.2 item 2; Table 1: F_C = 1, K = 1, G = I_C): depthwise
// convolution on the blocked layout.  The channel block is the vector dimension (G_b = C_b, Section 4.2.1): one
// thread owns four adjacent channels (a 128-bit lane), so a warp reads whole 128-byte lines.  The 3x3 kernel streams input rows
// through shared memory by TMA (padding supplied by the out-of-range zero fill) past threads that hold the sums of two
// neighbouring output columns (the paper's O_wb register tile); every input line leaves HBM once.  Other window shapes use the
// generic kernel (one output pixel per thread).
#include "common.cuh"
#include "sm100.cuh"
#include <string>
#include <unordered_map>

namespace small {

struct DwArgs {
    const float *in; const float *w; const float *bias; float *out;
    int H, W, FH, FW, S, pt, pl, OH, OW, C, CB;
    long long planes;
    bool relu;
};

__device__ __forceinline__ void fma4(float4 &a, const float4 &v, const float4 &w) {
    a.x = fmaf(v.x, w.x, a.x); a.y = fmaf(v.y, w.y, a.y); a.z = fmaf(v.z, w.z, a.z); a.w = fmaf(v.w, w.w, a.w);
}

// Generic window / stride: one output pixel x four channels per thread.
__global__ void __launch_bounds__(256) dwconv_generic_kernel(DwArgs a) {
    grid_dep_sync();
    grid_dep_trigger();
    const long long total = a.planes * a.OH * a.OW * 8;
    for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < total; t += (long long)gridDim.x * blockDim.x) {
        int q = (int)(t & 7);
        long long pix = t >> 3;
        int ow = (int)(pix % a.OW);
        long long r = pix / a.OW;
        int oh = (int)(r % a.OH);
        long long plane = r / a.OH;
        int cb = (int)(plane % a.CB);
        const float4 *src = reinterpret_cast<const float4 *>(a.in + plane * a.H * a.W * 32) + q;
        const float4 *wt = reinterpret_cast<const float4 *>(a.w + (size_t)cb * a.FH * a.FW * 32) + q;
        float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
        int cbase = cb * 32 + q * 4;
        if (a.bias) {   // bias has exactly C entries
            if (cbase + 0 < a.C) acc.x = a.bias[cbase + 0];
            if (cbase + 1 < a.C) acc.y = a.bias[cbase + 1];
            if (cbase + 2 < a.C) acc.z = a.bias[cbase + 2];
            if (cbase + 3 < a.C) acc.w = a.bias[cbase + 3];
        }
        int h0 = oh * a.S - a.pt, w0 = ow * a.S - a.pl;
        for (int x = 0; x < a.FH; ++x) {
            int h = h0 + x;
            if (h < 0 || h >= a.H) continue;
            for (int y = 0; y < a.FW; ++y) {
                int w = w0 + y;
                if (w < 0 || w >= a.W) continue;
                fma4(acc, src[(h * a.W + w) * 8], __ldg(wt + (x * a.FW + y) * 8));
            }
        }
        if (a.relu) {
            acc.x = acc.x > 0.f ? acc.x : 0.f; acc.y = acc.y > 0.f ? acc.y : 0.f;
            acc.z = acc.z > 0.f ? acc.z : 0.f; acc.w = acc.w > 0.f ? acc.w : 0.f;
        }
        reinterpret_cast<float4 *>(a.out)[t] = acc;
    }
}

// 3x3 window, stride ST (1 or 2): a stream of input rows through a ring of shared-memory slots, two persistent blocks per SM.
// A slot holds one input row of nn images (one channel block), as many as give the block's 32 column pairs work; wider rows
// are cut into bands of columns.  One warp fills the slots by TMA (padding is the out-of-range zero fill); eight warps
// compute, each waiting for rows and releasing them on its own.  Thread = (two neighbouring output columns, four channels):
// it reads each input row once (ST + 3 pixels) and adds it at once to the output rows that it belongs to, so two rows of
// sums are live instead of nine window pixels, in packed pairs of FMAs.  A block's work is one contiguous range of output rows
// (planes in order of channel block, then image: the filters change rarely), with 3 - ST more input rows where it begins
// inside a plane.  HBM bounds the large planes, filling the ring the small ones.  Measured, us, before (tiles with halos,
// double buffered, a barrier of the block per tile) and now: 128 x 64 channels on 56 x 56 45.8 / 42.2, 128 x 256 on 14 x 14
// 16.5 / 13.0, 128 x 512 on 7 x 7 12.3 / 10.1, 1024 x 64 on 25 x 5 18.5 / 16.3, 64 x 128 on 56 x 56 with stride 2 28.8 / 24.8.
constexpr int kDwWarps = 8, kDwThreads = (kDwWarps + 1) * 32, kDwPairs = kDwWarps * 4, kDwMaxSlots = 24;
struct Dw3Args {
    const float *w; const float *bias; float *out; int *status;
    int N, C, CB, OH, OW, pt, pl, Wb;
    int nn, groups;                        // images per row, and how many such sets
    int half, bands;                       // column pairs of an image in a band, bands of a row
    int share, extra;                      // output rows (channel blocks x groups x bands x OH) per block; the first `extra` have one more
    int slots;
    uint32_t slot_bytes;                   // nn x Wb pixels
    uint32_t wait_iters;                   // limit of the bounded waits (polls)
    bool relu;
};

__device__ __forceinline__ uint64_t dw_fma2(uint64_t a, uint64_t b, uint64_t c) {      // two FMAs
    uint64_t r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}

// A block's range as segments: some output rows of one channel block, set of images and band.
struct DwSegment {
    int left, cb, n, band, row, k;         // output rows left, channel block, first image, band, first row, rows
    __device__ __forceinline__ DwSegment(const Dw3Args &a) {
        const int b = (int)blockIdx.x, i0 = b * a.share + min(b, a.extra);
        left = a.share + (b < a.extra ? 1 : 0);
        int r = i0 / a.OH;
        row = i0 - r * a.OH;
        const int r2 = r / a.bands;
        band = r - r2 * a.bands;
        cb = r2 / a.groups; n = (r2 - cb * a.groups) * a.nn;
        k = min(a.OH - row, left);
    }
    __device__ __forceinline__ void next(const Dw3Args &a) {
        left -= k; row = 0;
        if (++band == a.bands) {
            band = 0; n += a.nn;
            if (n >= a.N) { n = 0; ++cb; }
        }
        k = min(a.OH, left);
    }
};

template <int ST>
__global__ void __launch_bounds__(kDwThreads, 2) dwconv3x3_tma_kernel(const __grid_constant__ CUtensorMap map_in, const Dw3Args a) {
    constexpr int kHalo = 3 - ST;          // input rows that an output row shares with the next
    constexpr int kPx = ST + 3;            // input pixels of a row under two outputs
    extern __shared__ uint8_t smem_raw[];
    const uint32_t base = (sm100::smem_u32(smem_raw) + 127u) & ~127u;
    __shared__ __align__(8) unsigned long long bars[2 * kDwMaxSlots];
    __shared__ int abort_flag;
    const uint32_t full = sm100::smem_u32(&bars[0]), empty = full + 8 * kDwMaxSlots;
    const int warp = sm100::warp_index();

    if (threadIdx.x < kDwMaxSlots) {
        sm100::mbar_init(full + 8 * threadIdx.x, 1);
        sm100::mbar_init(empty + 8 * threadIdx.x, kDwWarps);
        sm100::mbar_fence_init();
        if (threadIdx.x == 0) abort_flag = 0;
    }
    DwSegment t(a);
    __syncthreads();
    grid_dep_sync();
    grid_dep_trigger();
    int s = 0;
    if (warp == kDwWarps) {
        uint32_t par = 1;
        bool wrapped = false, alive = true;
        for (; t.left > 0 && alive; t.next(a)) {
            const int rows = t.k * ST + kHalo, h0 = t.row * ST - a.pt, w0 = t.band * a.half * 2 * ST - a.pl;
            for (int i = 0; i < rows; ++i) {
                if (wrapped) alive = sm100::mbar_wait_uniform(empty + 8 * s, par, &abort_flag, a.status, a.wait_iters);
                if (!alive) break;
                if (sm100::elect_one()) {
                    sm100::mbar_expect_tx(full + 8 * s, a.slot_bytes);
                    sm100::tma_load_5d(base + s * a.slot_bytes, &map_in, full + 8 * s, 0, w0, h0 + i, t.cb, t.n);
                }
                __syncwarp();
                if (++s == a.slots) { s = 0; par ^= 1; wrapped = true; }
            }
        }
        // after a timeout: give copies that may still be in flight a bounded grace period before the block exits
        if (!alive)
            for (uint32_t k = 0; k < (1u << 14); ++k) __nanosleep(200);
        return;
    }
    // the thread's place: image of the set, column pair, four channels (threads past the last pair keep its place and store nothing)
    const int q = threadIdx.x & 7, unit = threadIdx.x >> 3, last = a.nn * a.half - 1, p = min(unit, last);
    const int img = p / a.half, pair = p - img * a.half;
    const uint8_t *const mine = smem_raw + (base - sm100::smem_u32(smem_raw)) + (uint32_t)(img * a.Wb + pair * 2 * ST) * 128 + q * 16;
    uint32_t par = 0;
    int w_cb = -1, prev = -1;
    bool alive = true;
    ulonglong2 w[9], bias2 = make_ulonglong2(0ull, 0ull);
    ulonglong2 px[kPx], A[2], B[2];
    // The next input row.  Its slot is released at the row after it, so that no warp waits for its own loads to release it.  One
    // lane hands the slot back for the warp: the barrier in front of it puts the other lanes' reads of the slot before its arrival
    // (41.8 us with it and without, 64 channels on 56 x 56, batch 128).
    auto load = [&]() {
        alive = sm100::mbar_wait_uniform(full + 8 * s, par, &abort_flag, a.status, a.wait_iters);
        __syncwarp();
        if (prev >= 0 && (threadIdx.x & 31) == 0) sm100::mbar_arrive(empty + 8 * prev);
        const uint8_t *from = mine + s * a.slot_bytes;
#pragma unroll
        for (int y = 0; y < kPx; ++y) px[y] = *reinterpret_cast<const ulonglong2 *>(from + y * 128);
        prev = s;
        if (++s == a.slots) { s = 0; par ^= 1; }
    };
    auto mac = [&](ulonglong2 (&to)[2], const ulonglong2 &from0, const ulonglong2 &from1, int x) {      // + the window's row x
        to[0].x = dw_fma2(px[0].x, w[x * 3].x, from0.x); to[0].y = dw_fma2(px[0].y, w[x * 3].y, from0.y);
        to[1].x = dw_fma2(px[ST].x, w[x * 3].x, from1.x); to[1].y = dw_fma2(px[ST].y, w[x * 3].y, from1.y);
#pragma unroll
        for (int y = 1; y < 3; ++y) {
            to[0].x = dw_fma2(px[y].x, w[x * 3 + y].x, to[0].x); to[0].y = dw_fma2(px[y].y, w[x * 3 + y].y, to[0].y);
            to[1].x = dw_fma2(px[ST + y].x, w[x * 3 + y].x, to[1].x); to[1].y = dw_fma2(px[ST + y].y, w[x * 3 + y].y, to[1].y);
        }
    };
    for (; t.left > 0 && alive; t.next(a)) {
        if (t.cb != w_cb) {                        // the channel block's filters and bias
            w_cb = t.cb;
            const ulonglong2 *wt = reinterpret_cast<const ulonglong2 *>(a.w + (size_t)w_cb * 9 * 32) + q;
#pragma unroll
            for (int i = 0; i < 9; ++i) w[i] = __ldg(wt + i * 8);
            const int c = w_cb * 32 + q * 4;
            float b[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) b[e] = a.bias && c + e < a.C ? __ldg(a.bias + c + e) : 0.0f;   // bias has exactly C entries
            bias2.x = ((uint64_t)__float_as_uint(b[1]) << 32) | __float_as_uint(b[0]);
            bias2.y = ((uint64_t)__float_as_uint(b[3]) << 32) | __float_as_uint(b[2]);
        }
        const int ow = (t.band * a.half + pair) * 2, n = t.n + img;
        const bool one = unit <= last && n < a.N && ow < a.OW, two = one && ow + 1 < a.OW;
        float *dst = a.out + ((((size_t)n * a.CB + t.cb) * a.OH + t.row) * a.OW + ow) * 32 + q * 4;
        load();
        mac(A, bias2, bias2, 0);
        if (ST == 1) {
            load();
            mac(A, A[0], A[1], 1);
            mac(B, bias2, bias2, 0);
        }
#pragma unroll 1
        for (int i = 0; i < t.k && alive; ++i, dst += a.OW * 32) {
            if (ST == 2) { load(); mac(A, A[0], A[1], 1); }
            load();
            mac(A, A[0], A[1], 2);
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                float4 f = make_float4(__uint_as_float((uint32_t)A[c].x), __uint_as_float((uint32_t)(A[c].x >> 32)), __uint_as_float((uint32_t)A[c].y), __uint_as_float((uint32_t)(A[c].y >> 32)));
                if (a.relu) {
                    f.x = f.x > 0.f ? f.x : 0.f; f.y = f.y > 0.f ? f.y : 0.f;
                    f.z = f.z > 0.f ? f.z : 0.f; f.w = f.w > 0.f ? f.w : 0.f;
                }
                if (alive && (c == 0 ? one : two)) __stcs(reinterpret_cast<float4 *>(dst + c * 32), f);
            }
            if (ST == 1) { mac(A, B[0], B[1], 1); mac(B, bias2, bias2, 0); }
            else mac(A, bias2, bias2, 0);
        }
    }
    if (!alive)
        for (uint32_t k = 0; k < (1u << 14); ++k) __nanosleep(200);
}

// Rows and ring of the TMA kernel; false if there is too much to count (then the generic kernel runs).
static bool plan_dw3(const Geom &g, int sms, size_t max_smem, Dw3Args &a, unsigned &grid) {
    const int half = (g.OW + 1) / 2;
    a.bands = ceil_div(half, kDwPairs);
    a.half = ceil_div(half, a.bands);
    a.Wb = (2 * a.half - 1) * g.S + 3;             // at most 129 pixels
    a.nn = kDwPairs / a.half;
    if (a.nn > g.N) a.nn = g.N;
    a.groups = ceil_div(g.N, a.nn);
    a.nn = ceil_div(g.N, a.groups);
    const long long items = (long long)g.CB * a.groups * a.bands * g.OH;
    if (items > (1LL << 30)) return false;
    a.slot_bytes = (uint32_t)(a.nn * a.Wb * 128);
    grid = (unsigned)(items < 2LL * sms ? items : 2LL * sms);
    // the ring: at most half of the SM's shared memory, and no more than a block's rows
    a.share = (int)(items / grid); a.extra = (int)(items % grid);
    const int rows = (a.share + 1) * 3;
    a.slots = (int)(((max_smem + 1024) / 2 - 2048) / a.slot_bytes);
    if (a.slots > kDwMaxSlots) a.slots = kDwMaxSlots;
    if (a.slots > rows) a.slots = rows;
    return a.slots >= 3;
}

namespace {
typedef void (*DwKernel)(const CUtensorMap, const Dw3Args);
struct DwLaunch { CUtensorMap map; Dw3Args a; DwKernel kern; unsigned grid; size_t smem; };
typedef std::unordered_map<std::string, DwLaunch> DwCache;
}  // namespace

void free_dw_cache(small_ctx *ctx) {
    delete static_cast<DwCache *>(ctx->dw_cache);
    ctx->dw_cache = nullptr;
}

int launch_dwconv(small_ctx *ctx, const float *in, const float *w, const float *bias, float *out, const Geom &g, bool relu, cudaStream_t st) {
    if (g.FH == 3 && g.FW == 3 && (g.S == 1 || g.S == 2)) {
        std::string key;
        const int f[] = {g.N, g.C, g.H, g.W, g.S, g.pt, g.pb, g.pl, g.pr, relu ? 1 : 0, (int)ctx->wait_iters};
        const void *ptrs[] = {in, w, bias, out};
        key.append(reinterpret_cast<const char *>(f), sizeof(f));
        key.append(reinterpret_cast<const char *>(ptrs), sizeof(ptrs));
        if (!ctx->dw_cache) ctx->dw_cache = new DwCache();
        DwCache &cache = *static_cast<DwCache *>(ctx->dw_cache);
        auto it = cache.find(key);
        DwLaunch L{};
        Dw3Args &t = L.a;
        if (it == cache.end() && plan_dw3(g, ctx->sm_count, ctx->max_smem_optin, t, L.grid)) {
            t.w = w; t.bias = bias; t.out = out; t.status = ctx->dev_status; t.wait_iters = ctx->wait_iters;
            t.N = g.N; t.C = g.C; t.CB = g.CB; t.OH = g.OH; t.OW = g.OW; t.pt = g.pt; t.pl = g.pl; t.relu = relu;
            CUresult r = sm100::encode_blocked_map(ctx->encode_tiled, &L.map, in, g.N, g.CB, g.H, g.W, t.Wb, 1, t.nn);
            if (r != CUDA_SUCCESS) { ctx->last_cuda = (int)r; return SMALL_ERR_CUDA; }
            L.smem = t.slots * (size_t)t.slot_bytes + 128;
            L.kern = g.S == 1 ? dwconv3x3_tma_kernel<1> : dwconv3x3_tma_kernel<2>;
            cudaError_t e = cudaFuncSetAttribute(L.kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)ctx->max_smem_optin / 2);
            if (e != cudaSuccess) { ctx->last_cuda = (int)e; return SMALL_ERR_CUDA; }
            if (cache.size() >= 4096) cache.clear();
            it = cache.emplace(std::move(key), L).first;
        }
        if (it != cache.end()) {
            const DwLaunch &C = it->second;
            launch_kernel(ctx, C.kern, dim3(C.grid), dim3(kDwThreads), C.smem, st, C.map, C.a);
            return check_launch(ctx);
        }
    }
    DwArgs a{in, w, bias, out, g.H, g.W, g.FH, g.FW, g.S, g.pt, g.pl, g.OH, g.OW, g.C, g.CB, (long long)g.N * g.CB, relu};
    long long total = a.planes * g.OH * g.OW * 8;
    long long want = (total + 255) / 256, cap = (long long)ctx->sm_count * 32;
    int grid = (int)(want < cap ? want : cap);
    launch_kernel(ctx, dwconv_generic_kernel, dim3(grid), dim3(256), 0, st, a);
    return check_launch(ctx);
}

}  // namespace small
