// Host side of the resident network kernel (net_resident.cuh): which run of layers at the end of a list it takes, where the
// tensors lie in shared memory, how many thread blocks share an image, and the launch.
#include <algorithm>
#include <cstring>
#include <map>
#include <memory>
#include <unordered_map>
#include <vector>

#include "net_resident.cuh"

namespace small {

using namespace resident;

namespace {

struct Tensor { int C, H, W, pitch, size, off, last_use; bool external; int slot; };

uint32_t multiplier(int d) { return d <= 1 ? 0u : (uint32_t)((1ull << 32) / (unsigned)d) + 1u; }      // see quotient

int act_pitch(int C) { return ((C + 7) & ~7) + 4; }

// Can this layer run on chip?  `last`: it ends the list.
bool op_supported(const small_layer &L, int N, bool last, unsigned &math, Geom &g) {
    switch (L.op) {
        case SMALL_OP_CONV:
            if (make_geom(g, N, L.C, L.K, L.H, L.W, L.FH, L.FW, L.stride, L.pad_t, L.pad_b, L.pad_l, L.pad_r)) return false;
            // (fewer than 8 channels: a K step would be mostly padding, and such layers have a kernel of their own)
            if (L.C < 8 || L.C > 256 || L.K > 512 || L.FH * L.FW > 25 || L.FH * L.FW * ((L.C + 7) / 8) > kMaxSteps) return false;
            break;
        case SMALL_OP_DWCONV:
            if (make_geom(g, N, L.C, L.C, L.H, L.W, L.FH, L.FW, L.stride, L.pad_t, L.pad_b, L.pad_l, L.pad_r)) return false;
            return L.FH == 3 && L.FW == 3 && L.stride <= 2 && L.C <= 256;      // (filters and bias fit in one stage)
        case SMALL_OP_POOL:
            if (make_geom(g, N, L.C, L.C, L.H, L.W, L.FH, L.FW, L.stride, L.pad_t, L.pad_b, L.pad_l, L.pad_r)) return false;
            return !last && L.pool_mode == SMALL_POOL_AVG && L.FH == L.H && L.FW == L.W && L.C <= 512 && !(L.pad_t | L.pad_b | L.pad_l | L.pad_r);
        case SMALL_OP_FC:
            if (!last || L.C < 1 || L.C > 512 || L.K < 1 || L.K > 256) return false;
            break;
        default: return false;
    }
    const unsigned m = L.flags & SMALL_MATH_MASK;
    if (math == ~0u) math = m;
    return m == math;
}

struct Plan { Args a; size_t smem; int from; bool ok; int out_slot; int in_slot[kMaxInputs]; unsigned math; };

// Layers from .. n - 1 as one kernel; ok = false where they do not fit.
Plan plan_run(const small_layer *layers, int n, int from, int N, size_t max_smem, bool keep) {
    Plan p{};
    p.ok = false;
    p.from = from;
    // only runs that end in the classifier head: what a list ends in is a result, and a run's other tensors are not written
    if (n - from < 2 || n - from > kMaxOps || layers[n - 1].op != SMALL_OP_FC) return p;
    if (layers[from].op != SMALL_OP_CONV && layers[from].op != SMALL_OP_DWCONV) return p;      // the filter stream starts with the first operation
    unsigned math = ~0u;
    std::vector<Tensor> t;
    std::map<int, int> at;                               // slot -> tensor it holds
    struct Use { int src, dst; Geom g; };
    std::vector<Use> use;
    auto external = [&](int slot, int C, int H, int W) {
        t.push_back(Tensor{C, H, W, act_pitch(C), 0, 0, -1, true, slot});
        return at[slot] = (int)t.size() - 1;
    };
    Args &a = p.a;
    for (int i = from; i < n; ++i) {
        const small_layer &L = layers[i];
        Use u{};
        if (!op_supported(L, N, i == n - 1, math, u.g)) return p;
        if (L.op == SMALL_OP_POOL && (layers[i + 1].op != SMALL_OP_FC || layers[i + 1].src != L.dst || layers[i + 1].C != L.C)) return p;
        if (L.op == SMALL_OP_FC && (i == from || layers[i - 1].op != SMALL_OP_POOL)) return p;
        if (L.dst == SMALL_SLOT_OUTPUT && i != n - 1) return p;
        u.src = at.count(L.src) ? at[L.src] : external(L.src, L.C, L.H, L.W);
        if (t[u.src].C != L.C || t[u.src].H != L.H || t[u.src].W != L.W) return p;
        t[u.src].last_use = i;
        const int OH = L.op == SMALL_OP_FC ? 1 : u.g.OH, OW = L.op == SMALL_OP_FC ? 1 : u.g.OW, K = L.op == SMALL_OP_CONV || L.op == SMALL_OP_FC ? L.K : L.C;
        if (L.op == SMALL_OP_CONV && (L.flags & SMALL_ACCUMULATE)) {
            u.dst = at.count(L.dst) ? at[L.dst] : external(L.dst, K, OH, OW);
            if (t[u.dst].C != K || t[u.dst].H != OH || t[u.dst].W != OW) return p;
        } else {
            t.push_back(Tensor{K, OH, OW, act_pitch(K), 0, 0, -1, false, L.dst});
            u.dst = (int)t.size() - 1;
            at[L.dst] = u.dst;
        }
        t[u.dst].last_use = i;
        use.push_back(u);
    }
    int n_ext = 0;
    for (Tensor &x : t) {
        if ((long long)x.H * x.W * x.pitch > (1 << 20)) return p;
        x.size = (x.H * x.W * x.pitch + 3) & ~3;
        if (x.external && ++n_ext > kMaxInputs) return p;
    }
    // first fit; external tensors are loaded before the first operation
    const long long limit = (long long)(max_smem - 1024) / 4;
    struct Block { int off, size, tensor; };
    std::vector<Block> live;
    long long top = 0;
    auto place = [&](int ti) {
        long long off = 0;
        std::sort(live.begin(), live.end(), [](const Block &x, const Block &y) { return x.off < y.off; });
        for (const Block &b : live)
            if (off + t[ti].size > b.off) off = std::max(off, (long long)b.off + b.size);
            else break;
        t[ti].off = (int)off;
        live.push_back(Block{(int)off, t[ti].size, ti});
        top = std::max(top, off + t[ti].size);
    };
    a.zero = 0; a.ops = kZeroFloats; a.steps = a.ops + (int)(sizeof(a.op) / sizeof(float)); a.ring = a.steps + 2 * kMaxSteps; a.scratch = a.ring + kStages * kStageFloats;      // (scratch behind the ring: see mma_steps)
    live.push_back(Block{0, a.scratch + kScratchFloats, -1});
    for (int i = 0; i < (int)t.size(); ++i)
        if (t[i].external) {
            place(i);
            a.in[a.n_in] = Input{nullptr, t[i].C, t[i].H, t[i].W, t[i].off, t[i].pitch};
            p.in_slot[a.n_in++] = t[i].slot;
        }
    std::vector<Block> since;                            // what depthwise layers read since the last exchange
    for (int i = from; i < n; ++i) {
        const small_layer &L = layers[i];
        const Use &u = use[i - from];
        bool placed = false;
        for (const Block &b : live) placed = placed || b.tensor == u.dst;
        if (!placed && L.op != SMALL_OP_FC) place(u.dst);
        if (top > limit) return p;
        Op &o = a.op[a.n_ops++];
        o.kind = L.op == SMALL_OP_CONV ? kConv : L.op == SMALL_OP_DWCONV ? kDw : L.op == SMALL_OP_POOL ? kGap : kFc;
        o.C = L.C; o.K = t[u.dst].C; o.H = L.H; o.W = L.W; o.OH = t[u.dst].H; o.OW = t[u.dst].W;
        o.FH = L.FH; o.FW = L.FW; o.S = L.stride; o.pt = L.pad_t; o.pl = L.pad_l;
        o.src = t[u.src].off; o.sp = t[u.src].pitch; o.dst = t[u.dst].off; o.dp = t[u.dst].pitch;
        o.relu = (L.flags & SMALL_RELU) ? 1 : 0; o.accumulate = (L.flags & SMALL_ACCUMULATE) ? 1 : 0;
        o.w = L.w_blk; o.bias = L.bias;
        const int C4 = ((o.C + 7) & ~7) >> 2;
        o.by_ow = multiplier(o.OW); o.by_c4 = multiplier(C4); o.by_cols = multiplier(o.OW * C4);
        if (o.kind == kDw) {
            // runs of rows: as many as give every thread one, of at least two rows
            o.segs = std::max(1, std::min(kThreads / (o.OW * C4), (o.OH + 1) / 2));
            o.seg_rows = ceil_div(o.OH, o.segs);
            o.segs = ceil_div(o.OH, o.seg_rows);
        } else if (o.kind == kGap) {
            o.segs = std::min(std::min(kThreads / C4, kScratchFloats / (C4 * 4)), 32);      // groups of pixels
        }
        if (o.kind == kDw) since.push_back(Block{t[u.src].off, t[u.src].size, u.src});
        if (o.kind == kConv) {
            // the blocks of a cluster store into each other's copies of this output: where it takes the place of something a
            // slower block may still be reading, they meet before it
            for (const Block &b : since)
                if (t[u.dst].off < b.off + b.size && b.off < t[u.dst].off + t[u.dst].size) a.op[a.n_ops - 2].exchange = 1;
            since.clear();
        }
        // (what a depthwise layer read stays for one operation more where there is room, so that the convolution behind it does
        // not take its place)
        live.erase(std::remove_if(live.begin(), live.end(), [&](const Block &b) {
                       return b.tensor >= 0 && i < n - 1 && t[b.tensor].last_use + (keep && t[b.tensor].size < limit / 8 && layers[t[b.tensor].last_use].op == SMALL_OP_DWCONV ? 1 : 0) <= i;
                   }), live.end());
    }
    p.out_slot = layers[n - 1].dst;
    // an image's result must not land where another image's input is still to be read
    for (int i = 0; i < a.n_in; ++i)
        if (p.in_slot[i] == p.out_slot) return p;
    a.n_stream = a.n_ops - 2;
    a.N = N;
    p.smem = (size_t)top * 4;
    p.math = math;
    p.ok = true;
    return p;
}

Kernel kernel_of(unsigned math) {
    return math == SMALL_MATH_FP32 ? resident_kernel_fp32() : math == SMALL_MATH_TF32 ? resident_kernel_tf32() : resident_kernel_x3();
}

// How every convolution is split over the G blocks of an image and their warps, and the estimated cycles of one image.
double tile_ops(Args &a, unsigned math, int G) {
    double total = 3000.0;
    for (int i = 0; i < a.n_ops; ++i) {
        Op &o = a.op[i];
        const int P = o.OH * o.OW, T = o.FH * o.FW, CB = blocks_of(o.C), tail = (o.C - (CB - 1) * 32 + 7) & ~7;
        if (o.kind != kConv) {
            // a block computes these whole: about 20 (four channels of a pixel) per cycle; the head waits for memory
            total += o.kind == kDw ? (double)P * ((o.C + 3) / 4) / 12.0 + 500.0 : 1500.0;
            continue;
        }
        o.rows = T * ((CB - 1) * 32 + tail);
        const int Kr = o.K <= 8 ? 8 : o.K <= 16 ? 16 : blocks_of(o.K) * 32;        // filters padded to a part's widths
        double best = -1.0;
        Op pick = o;
        for (int parts = 1; parts <= G; parts *= 2) {
            if (Kr % parts || (Kr / parts) % 8 || (Kr / parts > 32 && (Kr / parts) % 32) || (Kr / parts < 32 && Kr / parts != 8 && Kr / parts != 16)) continue;
            Op c = o;
            c.n_parts = parts; c.n_w = Kr / parts;
            c.lg_parts = 0;
            while ((1 << c.lg_parts) < parts) ++c.lg_parts;
            const int pw = c.n_w < 32 ? c.n_w : 32, panels = c.n_w / pw;
            c.pitch = pw == 32 ? 40 : pw == 16 ? 24 : 8;
            c.chunk_rows = kStageFloats / (panels * c.pitch) & ~7;
            if (c.chunk_rows < 8) continue;
            if (c.chunk_rows > c.rows) c.chunk_rows = c.rows;
            c.panel = c.chunk_rows * c.pitch;
            c.chunks = ceil_div(c.rows, c.chunk_rows);
            const int m_parts = G / parts, F = ceil_div(P, 16);
            const double ksteps = c.rows / 8.0;
            auto consider = [&](int mf, int nf, int m_all, int n_units, double step, int part_floats) {
                Op d = c;
                d.mf = mf; d.nf = nf; d.m_units = ceil_div(m_all, m_parts); d.n_units = n_units; d.by_units = multiplier(n_units);
                const int units = d.m_units * n_units;
                d.rounds = ceil_div(units, kWarps);
                d.lg_split = 0;
                while (d.lg_split < 2 && (units << (d.lg_split + 1)) <= kWarps && units * ((2 << d.lg_split) - 1) * part_floats <= kScratchFloats) ++d.lg_split;
                d.split = 1 << d.lg_split;
                // a scheduler's warps of a round share its pipes; a lone warp waits out its own latencies
                const int per = ceil_div(units < kWarps ? units * d.split : kWarps, 4);
                const double pass = ceil_div((int)ksteps, d.split) * (step * per > 80.0 ? step * per : 80.0) + d.chunks * 150.0 + 500.0;
                const double stream = (double)d.chunks * d.chunk_rows * panels * pw * 4.0 / 30.0;        // bytes through the ring
                const double t = d.rounds * (pass > stream ? pass : stream) + (double)P * o.K * (math == SMALL_MATH_FP32 ? 1.0 : 0.4) * (G == 8 ? 0.35 : G == 4 ? 0.2 : G == 2 ? 0.1 : 0.0);      // and the exchange
                if (best < 0.0 || t < best) { best = t; pick = d; }
            };
            if (math == SMALL_MATH_FP32) {
                const int px = 8 * (32 / pw);
                for (int q = 1; q <= (panels % 2 == 0 ? 2 : 1); ++q) consider(1, q, ceil_div(P, px), panels / q, 64.0 * q + 60.0, q * 256);
            } else {
                const bool x3 = math == SMALL_MATH_3XTF32;
                static const int tiles[3][2] = {{1, 1}, {1, 2}, {2, 2}};
                for (auto &t : tiles)
                    if (t[1] <= c.n_w / 8)
                        consider(t[0], t[1], ceil_div(F, t[0]), c.n_w / 8 / t[1], t[0] * t[1] * (x3 ? 24.0 : 8.0) + 6.0 * t[1] + 8.0 * t[0] + 10.0, t[0] * t[1] * 128);
            }
        }
        if (best < 0.0) return -1.0;
        o = pick;
        total += best + (G > 1 ? 1000.0 : 200.0);
    }
    return total;
}

struct Entry { std::vector<unsigned char> key; std::unique_ptr<Plan> p; };      // no plan: the run is not taken
struct State {
    int clusters[3][4] = {};                             // resident clusters of 1, 2, 4, 8 blocks per math mode; 0: not asked yet
    std::unordered_multimap<size_t, Entry> plans;        // finished plans by a few words of (batch, layers); the key has all of them
};
State &state_of(small_ctx *ctx) {
    if (!ctx->resident_state) ctx->resident_state = new State();
    return *static_cast<State *>(ctx->resident_state);
}

int clusters_of(small_ctx *ctx, unsigned math, int lg) {
    State &s = state_of(ctx);
    int &c = s.clusters[math == SMALL_MATH_FP32 ? 0 : math == SMALL_MATH_TF32 ? 1 : 2][lg];
    if (c) return c;
    if (lg == 0) return c = ctx->sm_count;
    const Kernel k = kernel_of(math);
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(ctx->sm_count / (1 << lg) * (1 << lg)); cfg.blockDim = dim3(kThreads); cfg.dynamicSmemBytes = ctx->max_smem_optin - 1024;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 1u << lg; attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr; cfg.numAttrs = 1;
    cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)ctx->max_smem_optin - 1024);
    if (cudaOccupancyMaxActiveClusters(&c, k, &cfg) != cudaSuccess || c < 1) { cudaGetLastError(); c = 1; }
    return c;
}

// What comes here: in the tensor-core modes, networks with at most two depthwise / 1x1 pairs in a row (longer runs of pairs are
// sep_chain.cu's); in FP32, batches of some 30 images (128 channels on 25 x 5) to 100 (64 channels) and more, on one to four blocks per
// image: smaller ones are faster as launches (launches_beat_on_chip in net.cu).
// Where the run is faster on chip than layer by layer.  `one_round`: every image has its own thread blocks; with more images
// than that the layer kernels, which see the whole batch, win.  Measured called directly, us, layer by layer / on chip, on stacks of
// a 10 x 4 stem and n pairs of a depthwise and a 1x1 layer of C channels on 25 x 5 (the keyword-spotting network: C = 64, n = 4):
//   Tensor-core modes: what counts is a layer's work on an image, which one to eight SMs do with warp-level MMAs while the layer
//   kernels use block-level ones, and the exchange, which grows with G.  3xTF32: C = 48 batch 1 (G = 8) 44.0 / 36.9, 148 (G = 1)
//   58.4 / 41.6; C = 64 8 42.2 / 47.3, 18 (G = 4) 44.1 / 43.1, 74 (G = 2) 51.5 / 45.1, 148 57.6 / 47.1; C = 72 8 48.8 / 55.2, 148
//   70.8 / 93.4; C = 96 8 49.4 / 67.9, 37 56.2 / 61.5, 148 72.0 / 112.7; C = 128 148 82.7 / 139.4; TF32 C = 64 8 38.0 / 41.0, 24 40.2 /
//   43.3, 48 44.1 / 41.2, 148 52.3 / 41.1.  So 600,000 products per layer and image, 2.4 million times blocks (C = 64 at G = 4 is 2.05
//   million, C = 48 at G = 8 2.3).  The 700 KB of filters of the depthwise-separable network stream through every block; that
//   network stays with the layer kernels, which share them between images.
//   FP32: the layer kernels are as far from their peak as this one.  C = 64 batch 1 51.4 / 52.0, 37 70.3 / 53.5, 148 93.7 / 57.6;
//   C = 128 24 102.6 / 78.0, 74 128 / 91.6, 148 (G = 1) 166 / 176; depthwise-separable network (at most 590,000 products) 1 200 / 131,
//   64 308 / 213, 80 (G = 1) 356 / 333, 100 337 / 351, 148 376 / 380.  Filters are dealt to the blocks by halves of whole blocks of 32: C = 96 batch 18 77.9 / 64.9, but 37 (G = 2) 86.1 / 96.1, 148
//   119.6 / 139.4; C = 160, whose five blocks of filters all stay together, 1 67.8 / 119, 37 94.5 / 288, 148 168 / 478.  Without depthwise
//   layers nothing is computed without an exchange: residual network batch 1 (G = 8) 131 / 98, 12 132 / 105, 16 (G = 4) 125 / 124;
//   3xTF32 batch 1 66 / 73.
bool worth_it(const Args &a, unsigned math, int G, bool one_round) {
    if (!one_round) return false;
    size_t filters = 0;
    double most = 0.0;                                   // products of a layer and image
    int depthwise = 0, uneven = 0;                       // uneven: the most filters, in whole blocks, of layers where these are no power of two
    for (int i = 0; i < a.n_ops; ++i) {
        const Op &o = a.op[i];
        depthwise += o.kind == kDw ? 1 : 0;
        if (o.kind != kConv) continue;
        const int Kr = blocks_of(o.K) * 32;
        const size_t f = (size_t)o.C * o.K * o.FH * o.FW;
        filters += f * 4;
        most = std::max(most, (double)f * o.OH * o.OW);
        if (Kr & (Kr - 1)) uneven = std::max(uneven, Kr);
    }
    if (math != SMALL_MATH_FP32) return depthwise && filters <= 256 * 1024 && most <= 600e3 && most * G <= 2.4e6;
    if (uneven > 96 || (uneven && G < 4) || (G == 1 && most > 1e6)) return false;
    return depthwise || G == 8;
}

// The plan for layers from .. n - 1, nullptr where they do not run on chip.  Every call of a network asks, so what can be seen
// without a plan is answered first; plans are made once per batch and list (2 to 25 us each).
const Plan *find_plan(small_ctx *ctx, const small_layer *layers, int n, int from, int N) {
    if (N > ctx->sm_count || n - from < 2 || layers[n - 1].op != SMALL_OP_FC || layers[n - 2].op != SMALL_OP_POOL) return nullptr;
    if ((layers[n - 1].flags & SMALL_MATH_MASK) != SMALL_MATH_FP32) {
        int i = from;
        while (i < n && layers[i].op != SMALL_OP_DWCONV) ++i;
        if (i == n) return nullptr;
    }
    State &s = state_of(ctx);
    const int head[2] = {N, from};
    const size_t lb = sizeof(small_layer) * (size_t)n;
    const size_t words = ((size_t)N * 64 + from) * 64 + n + ((reinterpret_cast<size_t>(layers[n - 1].w_blk) ^ reinterpret_cast<size_t>(layers[0].w_blk)) << 16);
    const auto range = s.plans.equal_range(words);
    for (auto it = range.first; it != range.second; ++it) {
        const Entry &e = it->second;
        if (e.key.size() == lb + sizeof(head) && !memcmp(e.key.data(), head, sizeof(head)) && !memcmp(e.key.data() + sizeof(head), layers, lb)) return e.p.get();
    }
    Entry e;
    e.key.resize(lb + sizeof(head));
    memcpy(e.key.data(), head, sizeof(head));
    memcpy(e.key.data() + sizeof(head), layers, lb);
    Plan p{};
    p.ok = false;
    for (int s0 = from; s0 < n; ++s0) {
        p = plan_run(layers, n, s0, N, ctx->max_smem_optin, true);
        if (!p.ok) p = plan_run(layers, n, s0, N, ctx->max_smem_optin, false);
        if (p.ok) break;
    }
    if (p.ok) {
        Args &a = p.a;
        double best = 0.0;
        int best_g = 0;
        for (int lg = 0; lg < 4; ++lg) {
            const int c = clusters_of(ctx, p.math, lg);
            const double t = (double)ceil_div(N, c) * tile_ops(a, p.math, 1 << lg);
            if (t > 0.0 && (!best_g || t < best)) { best = t; best_g = 1 << lg; }
        }
        a.G = best_g;
        if (!best_g || !worth_it(a, p.math, best_g, N <= clusters_of(ctx, p.math, best_g == 8 ? 3 : best_g == 4 ? 2 : best_g - 1))) p.ok = false;
        else tile_ops(a, p.math, best_g);
    }
    if (p.ok) e.p.reset(new Plan(p));
    if (s.plans.size() >= 512) s.plans.clear();
    return s.plans.emplace(words, std::move(e))->second.p.get();
}

}  // namespace

void free_resident_state(small_ctx *ctx) {
    delete static_cast<State *>(ctx->resident_state);
    ctx->resident_state = nullptr;
}

int resident_from(small_ctx *ctx, const small_layer *layers, int n, int from, int N) {
    const Plan *p = find_plan(ctx, layers, n, from, N);
    return p ? p->from : -1;
}

int launch_resident(small_ctx *ctx, const small_layer *layers, int n, int from, int N, const std::function<const float *(int)> &rd,
                    const std::function<float *(int)> &wr, cudaStream_t st) {
    const Plan *p = find_plan(ctx, layers, n, from, N);
    if (!p) return SMALL_ERR_UNSUPPORTED;
    Args a = p->a;
    for (int i = 0; i < a.n_in; ++i) a.in[i].g = rd(p->in_slot[i]);
    a.out = wr(p->out_slot);
    const Kernel k = kernel_of(p->math);
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)ctx->max_smem_optin - 1024);
    if (e != cudaSuccess) { ctx->last_cuda = (int)e; return SMALL_ERR_CUDA; }
    int lg = 0;
    while ((1 << lg) < a.G) ++lg;
    const int clusters = std::min(N, clusters_of(ctx, p->math, lg));
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)(clusters * a.G)); cfg.blockDim = dim3(kThreads); cfg.dynamicSmemBytes = p->smem; cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)a.G; attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = ctx->dependent == 1 ? 2 : 1;      // (the filter stream starts in front of the wait)
    e = cudaLaunchKernelEx(&cfg, k, a);
    (void)e;                                             // picked up by check_launch through cudaGetLastError
    return check_launch(ctx);
}

}  // namespace small
