// Shared host-side declarations of the library: context, launch checks, argument validation.
#pragma once

#include <cuda_runtime.h>
#include <cstddef>
#include <cstdint>
#include <functional>

#include "small.h"

#define SMALL_CB 32          // channel block of the blocked layout (floats): one 128-byte line
#define SMALL_API extern "C" __attribute__((visibility("default")))

// A workspace that small_run_net_host was called on: its two input staging areas (see there).
struct small_host_stage {
    const char *base;        // nullptr: entry free
    size_t bytes;            // of the workspace that the calls use
    const char *in;          // the first staging area; the second one lies behind it
    size_t in_bytes;
    int next, used[2];       // area of the next call; whether an area was read yet
    int ordered;             // a call on this memory was captured: its replays read the first area at times unknown here
    void *ev_read[2];        // cudaEvent_t: the layer that read the area last has finished
    unsigned long long last; // call that used the entry last
};

struct small_ctx {
    int device;
    int last_cuda;           // last cudaError_t / CUresult seen
    int *dev_status;         // device status word (timeouts of bounded waits)
    void *encode_tiled;      // cuTensorMapEncodeTiled, resolved through the runtime
    int sm_count;
    size_t max_smem_optin;
    int overlap;             // layers are dependent launches, called on their own or by small_run_net (see launch_kernel)
    int dependent;           // how the next layer is launched: 0 the ordinary way, 1 and 2 as a dependent launch (see launch_kernel)
    int in_net;              // small_run_net is issuing layers: it sets `dependent`
    unsigned wait_iters;     // limit (polls) of every bounded device-side wait; small_set_wait_limit
    void *tc_cache;          // finished launches of the tensor-core kernel by (shape, mode, tensors); conv_tc.cu
    void *mma_cache;         // the same for the warp-level tensor-core kernel; conv_mma.cu
    void *resident_state;    // plans of the resident network kernel; net_resident.cu
    void *chain_state;       // plans and finished launches of runs of depthwise and 1x1 pairs; sep_chain.cu
    void *direct_cache;      // the same for the register-tiled FP32 kernel; conv_direct.cu
    void *dw_cache;          // the same for the depthwise 3x3 kernel; dwconv.cu
    void *thin_cache;        // the same for the kernel of few input channels; conv_thin.cu
    void *path_cache;        // kernel family per shape, mode and path setting; api.cu
    void *i8_cache;          // the same for the quantised convolution; conv_i8.cu
    void *static_workspace;  // device address of the library's built-in workspace array on this device (net_static.cu)
    int branch_overlap;      // small_run_net runs independent neighbouring layers side by side (side stream)
    void *side_stream, *ev_fork, *ev_join;   // cudaStream_t / cudaEvent_t of that
    void *copy_stream, *ev_h2d, *ev_start;   // small_run_net_host: input copies on their own stream
    small_host_stage host_stage[8];          // the workspaces it was called on latest
    unsigned long long host_calls;
    int host_ordered;        // an entry with `ordered` set had to make room: every copy keeps the caller's order from then on
    unsigned net_fusion;     // SMALL_FUSE_*: which neighbouring layers small_run_net runs as one fused layer
    int conv_path;           // SMALL_CONV_PATH_*: automatic, or one kernel family forced where it takes the shape
    int fc_chain_tile;       // images per thread block of the fused chain of full reductions: 0 = by batch size, else 32, 64 or 128
};

namespace small {

constexpr int kSmCount = 148;      // of a B200: for questions about a shape that are asked without a context

static inline int ceil_div(int a, int b) { return (a + b - 1) / b; }
static inline int blocks_of(int C) { return (C + SMALL_CB - 1) / SMALL_CB; }
static inline size_t packed_elems(int N, int C, int H, int W) {
    if (N < 1 || C < 1 || H < 1 || W < 1) return 0;
    return (size_t)N * blocks_of(C) * SMALL_CB * (size_t)H * W;
}
static inline int out_size(int I, int F, int S, int pa, int pb) {
    if (I < 1 || F < 1 || S < 1) return 0;
    int span = I + pa + pb - F;
    if (span < 0) return 0;
    return span / S + 1;
}
static inline bool aligned16(const void *p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }
static inline bool ranges_overlap(const void *a, size_t na, const void *b, size_t nb) {
    uintptr_t a0 = reinterpret_cast<uintptr_t>(a), b0 = reinterpret_cast<uintptr_t>(b);
    return a0 < b0 + nb && b0 < a0 + na;
}
static inline int check_launch(small_ctx *ctx) {
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) { ctx->last_cuda = (int)e; return SMALL_ERR_CUDA; }
    return SMALL_OK;
}

// Dependent launches.  Every layer kernel of this library executes grid_dep_sync() before its first access to global
// memory that an earlier kernel of the stream may have written (or may still read), and nothing it does before that
// touches such memory; it also executes grid_dep_trigger().  A kernel launched with programmatic stream serialisation
// may therefore start while the kernel in front of it in the stream is still draining: its blocks become resident as
// that kernel's blocks leave, set up their shared memory, barriers and tensor memory, and then wait at
// grid_dep_sync() until the earlier kernel has completed and its writes are visible.  Launched the ordinary way,
// both instructions do nothing.  Chains stay ordered: a kernel cannot complete before its own grid_dep_sync()
// returns, so completion of kernel i implies completion of every kernel before it.
// What a layer may do in front of grid_dep_sync() depends on the kernel before it.  Behind a layer of the same network
// (ctx->dependent = 1) it may read its filters and biases: no layer writes them, and everything older than the network is finished, since
// a network's first kernel triggers behind its wait and no later one starts before that trigger.  (Later ones may trigger first:
// fc_chain.cu does.)  Behind any other kernel of the stream (2: a call of its own, a
// network's first layer) it reads nothing: the kernel in front may be what writes the filters.  Kernels that read constants early
// take that as `late` and wait first.
#ifdef __CUDACC__
__device__ __forceinline__ void grid_dep_sync() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void grid_dep_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

template <typename... KArgs, typename... Args>
static inline void launch_kernel(small_ctx *ctx, void (*kern)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st,
                                 Args &&...args) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid; cfg.blockDim = block; cfg.dynamicSmemBytes = smem; cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = ctx->dependent ? 1 : 0;
    cudaError_t e = cudaLaunchKernelEx(&cfg, kern, static_cast<KArgs>(args)...);
    (void)e;   // picked up by check_launch through cudaGetLastError
}
#endif

// A layer called on its own: a dependent launch of the second kind where those are on.  (Inside a network the network decides.)
struct CallOfItsOwn {
    small_ctx *ctx;
    int before;
    explicit CallOfItsOwn(small_ctx *c) : ctx(c), before(c->dependent) { if (!c->in_net) c->dependent = c->overlap ? 2 : 0; }
    ~CallOfItsOwn() { ctx->dependent = before; }
};

// Geometry of one windowed layer, validated once on the host and passed to kernels by value.
struct Geom {
    int N, C, K, H, W, FH, FW, S, pt, pb, pl, pr, OH, OW;
    int CB, KB;   // channel blocks of input and output
};

// Fills g and returns SMALL_OK, or the status that describes what is wrong.
int make_geom(Geom &g, int N, int C, int K, int H, int W, int FH, int FW, int S, int pt, int pb, int pl, int pr);

void free_tc_cache(small_ctx *);             // conv_tc.cu
void free_mma_cache(small_ctx *);            // conv_mma.cu
void free_i8_cache(small_ctx *);             // conv_i8.cu
void free_direct_cache(small_ctx *);         // conv_direct.cu
void free_dw_cache(small_ctx *);             // dwconv.cu
void free_thin_cache(small_ctx *);           // conv_thin.cu
void free_resident_state(small_ctx *);       // net_resident.cu
void free_chain_state(small_ctx *);          // sep_chain.cu
int resolve_static_workspace(small_ctx *);   // net_static.cu; called by small_init with the context's device current

// ---- kernel launchers (each in its own .cu); all return a small_status ----
int launch_pack(small_ctx *, const float *nchw, float *blk, int N, int C, int H, int W, cudaStream_t);
int launch_unpack(small_ctx *, const float *blk, float *nchw, int N, int C, int H, int W, cudaStream_t);
int launch_pack_conv_weights(small_ctx *, const float *w, float *wb, int C, int K, int FH, int FW, unsigned math, cudaStream_t);
int launch_pack_dw_weights(small_ctx *, const float *w, float *wb, int C, int FH, int FW, cudaStream_t);
int launch_relu(small_ctx *, const float *in, float *out, size_t n, cudaStream_t);
int launch_add(small_ctx *, const float *a, const float *b, float *out, size_t n, bool relu, cudaStream_t);
int launch_scale_shift(small_ctx *, const float *in, const float *scale, const float *shift, float *out, int N, int C, int H, int W,
                       bool relu, cudaStream_t);
int launch_upsample_nearest(small_ctx *, const float *in, float *out, int N, int C, int H, int W, int f, cudaStream_t);
int launch_pool(small_ctx *, const float *in, float *out, int32_t *idx, const Geom &, int mode, cudaStream_t);
int launch_dwconv(small_ctx *, const float *in, const float *w, const float *bias, float *out, const Geom &, bool relu, cudaStream_t);
int launch_fc(small_ctx *, const float *in, const float *w, const float *bias, float *out, int N, int J, int K, bool relu, cudaStream_t);
// global average pool over the H x W plane and the full reduction behind it as one kernel; w as launch_fc takes it
int launch_gap_fc(small_ctx *, const float *in, const float *w, const float *bias, float *out, int N, int C, int H, int W, int K,
                  bool relu, cudaStream_t);
// span > 0: group convolution - filter block kb reads `span` channel blocks from that of its first group on
// (Kg filters per group, groups S_C channels apart); span = 0: full reduction over all channel blocks
int launch_conv_fp32(small_ctx *, const float *in, const float *w, const float *bias, float *out, const Geom &,
                     bool relu, bool accumulate, cudaStream_t, int span = 0, int Kg = 0, int S_C = 0);
// register-tiled FP32 kernel: windows 1 or 3 wide, strides 1 and 2 (group convolutions as launch_conv_fp32 takes them)
bool conv_direct_supported(const Geom &, int span = 0, int Kg = 0, int S_C = 0);
long long conv_direct_blocks(const Geom &, int sms);     // thread blocks its plan launches (0: shape not taken)
int launch_conv_direct(small_ctx *, const float *in, const float *w, const float *bias, float *out, const Geom &,
                       bool relu, bool accumulate, cudaStream_t, int span = 0, int Kg = 0, int S_C = 0);
// the same kernel with a 2 x 2 stride-2 max pool taken in its STORE phase: out is [N][K][OH/2][OW/2]
bool conv_direct_pool_supported(const Geom &);
int launch_conv_direct_pool(small_ctx *, const float *in, const float *w, const float *bias, float *out, const Geom &, bool relu, cudaStream_t);
// a run of 2 to 8 full reductions of width <= 128 as one tensor-core kernel (fc_chain.cu); widths has L + 1 entries
bool fc_chain_supported(const int *widths, int L, unsigned math);
int launch_fc_chain(small_ctx *, const float *in, const float *const *w_blk, const float *const *bias, const int *widths,
                    const int *relu, float *out, int L, int N, unsigned math, cudaStream_t);
// at most four input channels, 3 x 3 (strides 1, 2) or the 10 x 4 stride-2 window: FP32 FMAs with the filters in registers
bool conv_thin_supported(const Geom &);
// nchw_in: `in` is the NCHW tensor float[N][C][H][W] instead of the blocked one (used at a network's edge)
int launch_conv_thin(small_ctx *, const float *in, const float *w, const float *bias, float *out, const Geom &,
                     bool relu, bool accumulate, cudaStream_t, bool nchw_in = false);
int group_conv_span(int C, int F_C, int S_C, int Kg);      // channel blocks a filter block of a group convolution needs
int launch_pack_group_conv_weights(small_ctx *, const float *w, float *wb, int C, int F_C, int S_C, int Kg, int FH, int FW, cudaStream_t);
// tensor-core implicit GEMM; mode is SMALL_MATH_TF32 or SMALL_MATH_3XTF32
// x3: with the doubled stages of 3xTF32.  groups > 1: a group convolution whose groups are whole channel blocks; the
// Geom then holds one group's channels (C = F_C) and all filters (K = groups x filters per group).
// A depthwise 3x3 fused in front of a 1x1 convolution: the Geom given to the two functions below is the 1x1 layer over
// the depthwise output (H = W = that output's size); this describes the depthwise layer and its input.
struct DwFuse { const float *w; const float *bias; int C, H, W, s, pt, pl, relu; };
bool conv_tc_supported(const Geom &, bool x3 = false, int groups = 1, const DwFuse *dw = nullptr);
int launch_conv_tc(small_ctx *, const float *in, const float *w_hi, const float *w_lo, const float *bias, float *out,
                   const Geom &, bool relu, bool accumulate, unsigned mode, cudaStream_t, int groups = 1, const DwFuse *dw = nullptr);
// warp-level tensor-core kernel (conv_mma.cu): one channel block, filters in tiles of 32, strides 1 and 2; reads the same
// filter sections as launch_conv_tc
bool conv_mma_supported(const Geom &, bool x3);
int launch_conv_mma(small_ctx *, const float *in, const float *w_hi, const float *w_lo, const float *bias, float *out,
                    const Geom &, bool relu, bool accumulate, unsigned mode, cudaStream_t);
// A 1x1 layer without padding and activation whose result a layer of few pixels is added to (a residual stage's shortcut); g: that layer
struct Shortcut { const float *in, *w, *w_hi, *w_lo, *bias; Geom g; };
// warp-level tensor-core kernel for few pixels (conv_split.cu), whose rule says where it is the fastest of the tensor-core kernels;
// any channels, filters, window and stride; reads the same filter sections
bool conv_split_preferred(const Geom &, bool x3, bool warp_level, int sms);     // warp_level: instead of conv_mma.cu, else conv_tc.cu
int launch_conv_split(small_ctx *, const float *in, const float *w_hi, const float *w_lo, const float *bias, float *out,
                      const Geom &, bool relu, bool accumulate, unsigned mode, cudaStream_t, const Shortcut * = nullptr);
// FP32 kernel for few pixels (conv_split_fp32.cu): the same for the layers that the other FP32 kernels would take
double conv_split_fp32_us(const Geom &, int sms);          // the time expected, 0 where another kernel is preferred
int launch_conv_split_fp32(small_ctx *, const float *in, const float *w, const float *bias, float *out, const Geom &,
                           bool relu, bool accumulate, cudaStream_t, const Shortcut * = nullptr);
// whether a layer called on its own (with a 32-byte aligned output) computes in FP32 under this math mode (api.cu)
bool conv_in_fp32(small_ctx *, const Geom &, unsigned math);
// a shortcut and the layer that is added to it as one launch of those kernels: whether they run there, and the launch (api.cu)
bool joined_split(small_ctx *, const Geom &shortcut, const Geom &, unsigned math, bool out_aligned32);
int launch_joined(small_ctx *, Shortcut, const float *in, const float *w, const float *bias, float *out, const Geom &, bool relu, unsigned math, cudaStream_t);
// a depthwise 3x3 and the 1x1 layer behind it as that kernel: the time expected (0: not taken), and the launch; gd / gp: the two layers
double split_pair_us(const Geom &gp, int sms);
int launch_split_pair(small_ctx *, const float *in, const float *dw, const float *dw_bias, bool dw_relu, const float *w, const float *bias,
                      float *out, const Geom &gd, const Geom &gp, bool relu, cudaStream_t);
// a run of layers up to the end of the list as one kernel (net_resident.cu): the first layer of the run at or behind `from`
// (-1: none), and its launch, which reads and writes whole tensors through rd / wr (slot -> address)
int resident_from(small_ctx *, const small_layer *layers, int n, int from, int N);
int launch_resident(small_ctx *, const small_layer *layers, int n, int from, int N, const std::function<const float *(int)> &rd,
                    const std::function<float *(int)> &wr, cudaStream_t);
// no layer from `from` on reads the slot before it is written again (net.cu)
bool slot_dead_after(const small_layer *layers, int n_layers, int from, int slot);
// a run of depthwise 3x3 -> 1x1 pairs as one kernel (sep_chain.cu): how many layers the run at layer i covers (0: none), with a
// global average pool and full reduction behind it where it ends in those, and its launch
int sep_chain_layers(small_ctx *, const small_layer *layers, int n, int i, int N);
int launch_sep_chain(small_ctx *, const small_layer *layers, int n, int i, int N, const float *in, float *out, cudaStream_t);
// quantised full channel reduction (conv_i8.cu): windows 1 or 3 wide, strides 1 and 2; w: [CB][FH*FW][KB*32][32] bytes,
// w_sums: [K][FH*FW] sums of weight bytes over the channels
int launch_q_conv(small_ctx *, const uint8_t *in, const uint8_t *w, const int *w_sums, const int *bias, uint8_t *out, const Geom &,
                  bool relu, int zx, int zw, int zo, int mult, int shift, cudaStream_t);
// tensor-core filter sections of a group convolution: [F_C/32][FH*FW][G*K][32 ci], TF32 part and residual
size_t group_conv_w_tc_elems(int F_C, int K, int G, int FH, int FW);
int launch_pack_group_conv_weights_tc(small_ctx *, const float *w, float *hi, float *lo, int F_C, int K, int G, int FH, int FW, cudaStream_t);

// Sizes (in floats) of the sections of a packed convolution filter buffer.
size_t conv_w_fp32_elems(int C, int K, int FH, int FW);   // [KB][CB][FH][FW][32 ci][32 ko]
size_t conv_w_tc_elems(int C, int K, int FH, int FW);     // [CB][FH*FW][KB*32][32 ci]

}  // namespace small
