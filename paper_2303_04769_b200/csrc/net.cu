// Networks: a list of layer descriptors run in order over caller-provided slots of one workspace (paper Section 5.3:
// layers share intermediate buffers; Section 4.4: every layer reads and writes the same layout, so nothing is
// reformatted between layers).
#include <vector>

#include "common.cuh"

namespace small {

struct SlotPlan {
    std::vector<size_t> bytes;    // per slot
    std::vector<size_t> offset;   // per slot, 256-byte aligned
    size_t total = 0;
    size_t in_bytes = 0, out_bytes = 0;      // of the network's input and output, as far as layers reach
};

static size_t round256(size_t b) { return (b + 255) & ~(size_t)255; }

// Output shape of a layer; false if the descriptor is malformed.
static bool layer_out_shape(const small_layer &L, int N, int &oc, int &oh, int &ow) {
    Geom g;
    switch (L.op) {
        case SMALL_OP_CONV:
            if (make_geom(g, N, L.C, L.K, L.H, L.W, L.FH, L.FW, L.stride, L.pad_t, L.pad_b, L.pad_l, L.pad_r)) return false;
            oc = L.K; oh = g.OH; ow = g.OW; return true;
        case SMALL_OP_DWCONV:
        case SMALL_OP_POOL:
            if (make_geom(g, N, L.C, L.C, L.H, L.W, L.FH, L.FW, L.stride, L.pad_t, L.pad_b, L.pad_l, L.pad_r)) return false;
            oc = L.C; oh = g.OH; ow = g.OW; return true;
        case SMALL_OP_RELU:
        case SMALL_OP_ADD:
            if (L.C < 1 || L.H < 1 || L.W < 1) return false;
            oc = L.C; oh = L.H; ow = L.W; return true;
        case SMALL_OP_FC:
            if (L.C < 1 || L.K < 1 || L.H != 1 || L.W != 1) return false;
            oc = L.K; oh = 1; ow = 1; return true;
        case SMALL_OP_DWPW:
            if (L.K < 1 || make_geom(g, N, L.C, L.C, L.H, L.W, 3, 3, L.stride, L.pad_t, L.pad_b, L.pad_l, L.pad_r)) return false;
            oc = L.K; oh = g.OH; ow = g.OW; return true;
        case SMALL_OP_CONVPOOL:
            if (make_geom(g, N, L.C, L.K, L.H, L.W, L.FH, L.FW, L.stride, L.pad_t, L.pad_b, L.pad_l, L.pad_r)) return false;
            if (g.OH < 2 || g.OW < 2) return false;
            oc = L.K; oh = g.OH / 2; ow = g.OW / 2; return true;
        default: return false;
    }
}

static bool plan_slots(const small_layer *layers, int n_layers, int N, SlotPlan &plan) {
    if (!layers || n_layers < 1 || N < 1) return false;
    auto need = [&](int slot, size_t bytes) {
        if (slot < 0) {
            size_t &most = slot == SMALL_SLOT_INPUT ? plan.in_bytes : plan.out_bytes;
            if (most < bytes) most = bytes;
            return slot == SMALL_SLOT_INPUT || slot == SMALL_SLOT_OUTPUT;
        }
        if (slot > 4096) return false;
        if ((size_t)slot >= plan.bytes.size()) plan.bytes.resize(slot + 1, 0);
        if (plan.bytes[slot] < bytes) plan.bytes[slot] = bytes;
        return true;
    };
    for (int i = 0; i < n_layers; ++i) {
        const small_layer &L = layers[i];
        int oc, oh, ow;
        if (!layer_out_shape(L, N, oc, oh, ow)) return false;
        size_t in_b = sizeof(float) * packed_elems(N, L.C, L.H, L.W), out_b = sizeof(float) * packed_elems(N, oc, oh, ow);
        if (!need(L.src, in_b) || !need(L.dst, out_b)) return false;
        if (L.op == SMALL_OP_ADD && !need(L.src2, in_b)) return false;
        if (L.dst == SMALL_SLOT_INPUT) return false;
    }
    plan.offset.resize(plan.bytes.size());
    size_t off = 0;
    for (size_t s = 0; s < plan.bytes.size(); ++s) { plan.offset[s] = off; off += round256(plan.bytes[s]); }
    plan.total = off;
    return true;
}

// ---- abstract fused layers (Section 6) chosen by the runner itself: the caller describes plain layers.
// A layer's result may stay on chip when the next layer is its only reader: nothing after that reads the slot before
// it is written again, and the pair's output slot is not the pair's input slot.
bool slot_dead_after(const small_layer *layers, int n_layers, int from, int slot) {
    for (int j = from; j < n_layers; ++j) {
        const small_layer &L = layers[j];
        if (L.src == slot || (L.op == SMALL_OP_ADD && L.src2 == slot)) return false;
        if (L.dst == slot) return !((L.flags & SMALL_ACCUMULATE) && L.op == SMALL_OP_CONV);
    }
    return true;
}

// Fusing a depthwise 3x3 with the 1x1 convolution behind it: one launch instead of two, but the fused kernel has eight depthwise
// warps per SM and half the strips, where the two kernels have whole SMs.  Measured called directly, us, separate / fused:
//   3xTF32, single pairs, batch 1: 64 channels on 56 x 56 12.2 / 10.4, 128 on 28 x 28 14.6 / 12.4, 256 on 14 x 14 20.5 / 18.6, but 64 on
//   14 x 14 10.5 / 10.4, on 7 x 7 7.2 / 9.4, keyword-spotting network 42 / 48: it pays from some 50,000 values per image on, and for
//   one channel block between other layers: depthwise-separable network none / its four pairs of at most 32 channels / all fused,
//   batch 1 125.8 / 124.2 / 126.0, 2 126.1 / 121.9 / 125.1, 3 129.6 / 122.8 / 126.7, 4 129.6 / 123.7 / 128.6.
//   TF32, where the two kernels are shorter: 64 on 56 x 56 10.4 / 10.4 (batch 4 11.6 / 12.4), 128 on 28 x 28 12.5 / 12.4, 256 on 14 x 14
//   13.5 / 16.5; networks of small layers take the same time and half of the host's, depthwise-separable batch 1 110.7 / 111.8, 2 110.0 /
//   109.9, 3 114.3 / 113.9, 4 115.2 / 114.2, 8 118.0 / 121.5 (host 65 / 39; replayed from a graph fused is 3 % behind): up to 20,000 values.
//   512 channels on 7 x 7 18.6 / 34.3 and 14.5 / 28.8: a block streams the filters of all 16 channel blocks.
static const int kFuseDwpwMaxImages = 4, kFuseDwpwMaxChannels = 256;
static const size_t kFuseDwpwMaxBytes = 1u << 20;      // of the intermediate tensor
static bool dwpw_pays(int N, int C, int K, int OH, int OW, unsigned math) {
    if (N > kFuseDwpwMaxImages || C > kFuseDwpwMaxChannels || K > kFuseDwpwMaxChannels || sizeof(float) * packed_elems(N, C, OH, OW) > kFuseDwpwMaxBytes) return false;
    const long long values = (long long)C * OH * OW;
    return math == SMALL_MATH_3XTF32 ? C <= 32 || values >= 50000 : values <= 20000;
}

// Two layers may run at the same time when neither writes a tensor the other one reads or writes.
static bool independent(const small_layer &A, const small_layer &Bn) {
    auto reads = [](const small_layer &L, int slot) {
        return L.src == slot || (L.op == SMALL_OP_ADD && L.src2 == slot) || ((L.flags & SMALL_ACCUMULATE) && L.op == SMALL_OP_CONV && L.dst == slot);
    };
    if (A.dst == Bn.dst || reads(Bn, A.dst) || reads(A, Bn.dst)) return false;
    return A.dst != SMALL_SLOT_INPUT && Bn.dst != SMALL_SLOT_INPUT;
}

// 0: layer i runs on its own; SMALL_OP_DWPW / SMALL_OP_CONVPOOL / kFusedPoolFc: layers i and i + 1 run as that fused layer
static const int kFusedPoolFc = 1000;      // (no descriptor op of its own: only the runner forms this pair)
static int fused_pair(const small_ctx *ctx, const small_layer *layers, int n_layers, int i, int N) {
    if (i + 1 >= n_layers) return 0;
    const small_layer &A = layers[i], &Bn = layers[i + 1];
    if (A.dst < 0 || Bn.src != A.dst || Bn.dst == A.src || Bn.dst == A.dst) return 0;
    if (!slot_dead_after(layers, n_layers, i + 2, A.dst)) return 0;
    Geom g;
    if (A.op == SMALL_OP_DWCONV && Bn.op == SMALL_OP_CONV && (ctx->net_fusion & (SMALL_FUSE_DWPW | SMALL_FUSE_DWPW_ALWAYS))) {
        const unsigned math = Bn.flags & SMALL_MATH_MASK;
        if (A.FH != 3 || A.FW != 3 || Bn.FH != 1 || Bn.FW != 1 || Bn.stride != 1 || (Bn.pad_t | Bn.pad_b | Bn.pad_l | Bn.pad_r)) return 0;
        if ((Bn.flags & SMALL_ACCUMULATE) || Bn.C != A.C || math == SMALL_MATH_FP32) return 0;
        if (make_geom(g, N, A.C, A.C, A.H, A.W, 3, 3, A.stride, A.pad_t, A.pad_b, A.pad_l, A.pad_r)) return 0;
        if (Bn.H != g.OH || Bn.W != g.OW) return 0;
        if (!(ctx->net_fusion & SMALL_FUSE_DWPW_ALWAYS) && !dwpw_pays(N, A.C, Bn.K, g.OH, g.OW, math)) return 0;
        return small_dwpw_fused(N, A.C, Bn.K, A.H, A.W, A.stride, A.pad_t, A.pad_b, A.pad_l, A.pad_r, math) ? SMALL_OP_DWPW : 0;
    }
    if (A.op == SMALL_OP_CONV && Bn.op == SMALL_OP_POOL && (ctx->net_fusion & SMALL_FUSE_CONVPOOL)) {
        if ((A.flags & SMALL_ACCUMULATE) || Bn.pool_mode != SMALL_POOL_MAX || Bn.FH != 2 || Bn.FW != 2 || Bn.stride != 2 ||
            (Bn.pad_t | Bn.pad_b | Bn.pad_l | Bn.pad_r) || Bn.C != A.K)
            return 0;
        if (make_geom(g, N, A.C, A.K, A.H, A.W, A.FH, A.FW, A.stride, A.pad_t, A.pad_b, A.pad_l, A.pad_r)) return 0;
        if (Bn.H != g.OH || Bn.W != g.OW) return 0;
        return small_conv_maxpool_fused(N, A.C, A.K, A.H, A.W, A.FH, A.FW, A.stride, A.pad_t, A.pad_b, A.pad_l, A.pad_r) ? SMALL_OP_CONVPOOL : 0;
    }
    if (A.op == SMALL_OP_POOL && Bn.op == SMALL_OP_FC && (ctx->net_fusion & SMALL_FUSE_POOLFC)) {
        // a global average pool (window = plane, no padding) and the full reduction over its channels
        if (A.pool_mode != SMALL_POOL_AVG || A.FH != A.H || A.FW != A.W || (A.pad_t | A.pad_b | A.pad_l | A.pad_r) || Bn.C != A.C) return 0;
        return small_gap_fc_fused(N, A.C, Bn.K, Bn.flags & SMALL_MATH_MASK) ? kFusedPoolFc : 0;
    }
    return 0;
}

// Length of the run of full reductions starting at layer i that runs as one fused kernel (0: none): each layer reads what
// the one before it wrote, nothing else reads those intermediates, every width between two layers is at most 128, one
// tensor-core math mode.
static int fc_chain_len(const small_ctx *ctx, const small_layer *layers, int n_layers, int i, int N, int *widths) {
    if (!(ctx->net_fusion & SMALL_FUSE_FC_CHAIN) || layers[i].op != SMALL_OP_FC) return 0;
    const unsigned math = layers[i].flags & SMALL_MATH_MASK;
    if (math != SMALL_MATH_TF32 && math != SMALL_MATH_3XTF32) return 0;
    if (layers[i].C > 8192 || layers[i].K > 128) return 0;       // the first layer's input may be wide, and the last one's output
    int L = 1;
    widths[0] = layers[i].C; widths[1] = layers[i].K;
    while (i + L < n_layers && L < 12) {
        const small_layer &P = layers[i + L - 1], &Q = layers[i + L];
        if (Q.op != SMALL_OP_FC || Q.src != P.dst || P.dst < 0 || (Q.flags & SMALL_MATH_MASK) != math || Q.C != P.K || Q.K > 1024 || P.K > 128) break;
        if (!slot_dead_after(layers, n_layers, i + L + 1, P.dst)) break;
        if (Q.dst == layers[i].src) break;                      // the run's output must not land on its input
        widths[L + 1] = Q.K;
        ++L;
    }
    (void)N;
    return L >= 2 ? L : 0;
}

// Layers i and i + 1 as a depthwise 3x3 and a 1x1 layer in FP32 that run as one launch (conv_split_fp32.cu): the time expected, 0 where
// they do not.
static double split_pair(const small_ctx *ctx, const small_layer *layers, int n_layers, int i, int N, Geom &gd, Geom &gp) {
    if (i + 1 >= n_layers) return 0.0;
    const small_layer &A = layers[i], &Bn = layers[i + 1];
    if (A.op != SMALL_OP_DWCONV || Bn.op != SMALL_OP_CONV || A.FH != 3 || A.FW != 3 || Bn.FH != 1 || Bn.FW != 1 || Bn.stride != 1 ||
        (Bn.pad_t | Bn.pad_b | Bn.pad_l | Bn.pad_r) || (Bn.flags & (SMALL_ACCUMULATE | SMALL_MATH_MASK)) || Bn.C != A.C)
        return 0.0;
    if (A.dst < 0 || Bn.src != A.dst || Bn.dst == A.src || Bn.dst == A.dst || !slot_dead_after(layers, n_layers, i + 2, A.dst)) return 0.0;
    if (make_geom(gd, N, A.C, A.C, A.H, A.W, 3, 3, A.stride, A.pad_t, A.pad_b, A.pad_l, A.pad_r)) return 0.0;
    if (Bn.H != gd.OH || Bn.W != gd.OW || make_geom(gp, N, A.C, Bn.K, gd.OH, gd.OW, 1, 1, 1, 0, 0, 0, 0)) return 0.0;
    return split_pair_us(gp, ctx->sm_count);
}

// Layers i and i + 1 as a residual stage's shortcut - 1x1, no padding, no activation - and the convolution that is added to its result.
static bool shortcut_pair(const small_layer *layers, int n_layers, int i, int N, Geom &sc, Geom &g) {
    if (i + 1 >= n_layers) return false;
    const small_layer &A = layers[i], &Bn = layers[i + 1];
    if (A.op != SMALL_OP_CONV || Bn.op != SMALL_OP_CONV || A.FH != 1 || A.FW != 1 || (A.pad_t | A.pad_b | A.pad_l | A.pad_r) || A.dst != Bn.dst || A.K != Bn.K ||
        (A.flags & (SMALL_RELU | SMALL_ACCUMULATE)) || !(Bn.flags & SMALL_ACCUMULATE) || (A.flags & SMALL_MATH_MASK) != (Bn.flags & SMALL_MATH_MASK))
        return false;
    if (make_geom(sc, N, A.C, A.K, A.H, A.W, 1, 1, A.stride, 0, 0, 0, 0)) return false;
    if (make_geom(g, N, Bn.C, Bn.K, Bn.H, Bn.W, Bn.FH, Bn.FW, Bn.stride, Bn.pad_t, Bn.pad_b, Bn.pad_l, Bn.pad_r)) return false;
    return sc.OH == g.OH && sc.OW == g.OW;
}

// A run that could stay on chip in FP32 (net_resident.cu), launch by launch instead: whether that is the faster form
// for its batch.  An operation costs the on-chip kernel 4.3 to 6.7 us whatever the batch - barriers, filters passing by - and the kernels
// of few pixels 2 to 9, growing with it.  us, on chip against launches: stem and two pairs of 64 channels on 25 x 5, batch 1 / 18 / 74 31.5 /
// 29.5 / 31.2 against 13.4 / 19.7 / 29.1; the keyword-spotting network (four pairs) 1 / 37 / 64 / 128 47.9 / 50.1 / 51.0 / 53.7 against 20.8 /
// 35.6 / 48.3 / 82; depthwise-separable network 1 / 16 / 64 115.7 / 142 / 208 against 55.8 / 94 / 164.  Without depthwise layers, where
// every operation ends in an exchange, it is 9 us and more (residual network 98 at batch 1 to 105 at 12).
static bool launches_beat_on_chip(const small_ctx *ctx, const small_layer *layers, int n_layers, int from, int N) {
    double us = 4.0;                              // the average pool and the classifier
    bool depthwise = false;
    for (int i = from; i + 2 < n_layers; ++i) {
        Geom g, gp;
        const small_layer &L = layers[i];
        depthwise |= L.op == SMALL_OP_DWCONV;
        if (const double t = split_pair(ctx, layers, n_layers, i, N, g, gp)) { us += t; ++i; continue; }
        if ((L.op != SMALL_OP_CONV && L.op != SMALL_OP_DWCONV) || make_geom(g, N, L.C, L.K, L.H, L.W, L.FH, L.FW, L.stride, L.pad_t, L.pad_b, L.pad_l, L.pad_r)) return false;
        const double out = (double)N * g.OH * g.OW * L.K;
        if (L.op == SMALL_OP_DWCONV) us += 2.5 + (out + (double)N * L.C * L.H * L.W) / 1e6;
        else if (const double t = conv_split_fp32_us(g, ctx->sm_count)) us += t;
        else us += 5.0 + (0.07 + out / 15e6) * L.C * L.FH * L.FW;
    }
    return us < (depthwise ? 4.5 : 9.0) * (n_layers - from);
}

// Do the network's input, its output and the slots lie apart?  Then tensors overlap only where they share a slot, which the forms of
// several layers look at.  Where the caller's tensors meet - an output over the input, say, which is no longer read by then - the layers are
// called one by one: each compares the addresses it is given.
static bool tensors_apart(const SlotPlan &plan, const void *in, const void *out, const void *slots) {
    return !ranges_overlap(in, plan.in_bytes, out, plan.out_bytes) && !ranges_overlap(in, plan.in_bytes, slots, plan.total) &&
           !ranges_overlap(out, plan.out_bytes, slots, plan.total);
}

// Runs of layers are kept on chip as one kernel where every kind of fusion is on.
static bool runs_allowed(const small_ctx *ctx) {
    const unsigned rest = SMALL_FUSE_CONVPOOL | SMALL_FUSE_FC_CHAIN | SMALL_FUSE_POOLFC;
    return (ctx->net_fusion & rest) == rest && (ctx->net_fusion & (SMALL_FUSE_DWPW | SMALL_FUSE_DWPW_ALWAYS)) && ctx->conv_path == SMALL_CONV_PATH_AUTO;
}

// How the runner takes the layers of a list, decided from the list, the batch, the context's settings and whether the caller's tensors lie
// apart (`apart`) and the output is 32-byte aligned (`out32`; slots are).
struct Forms {
    bool apart, out32, runs;
    int chain = -1, chain_layers = 0, on_chip = -1;      // a run of depthwise / 1x1 pairs (sep_chain.cu); without one, a run up to the end of the list (net_resident.cu)
    Forms(small_ctx *ctx, const small_layer *layers, int n_layers, int from, int N, bool apart, bool out32) : apart(apart), out32(out32), runs(apart && runs_allowed(ctx)) {
        if (!runs) return;
        for (int i = from; i < n_layers && !chain_layers; ++i)
            if ((chain_layers = sep_chain_layers(ctx, layers, n_layers, i, N)) > 0) chain = i;
        if (!chain_layers) on_chip = resident_from(ctx, layers, n_layers, from, N);
        if (on_chip >= 0 && (layers[n_layers - 1].flags & SMALL_MATH_MASK) == SMALL_MATH_FP32 && launches_beat_on_chip(ctx, layers, n_layers, on_chip, N)) on_chip = -1;
    }
    bool aligned(int slot) const { return slot >= 0 || out32; }
    // a shortcut and the layer that is added to it, where both are split over warps, as one launch
    bool joins(small_ctx *ctx, const small_layer *layers, int n_layers, int i, int N, Geom &sc, Geom &g) const {
        return runs && i + 1 != chain && i + 1 != on_chip && shortcut_pair(layers, n_layers, i, N, sc, g) &&
               joined_split(ctx, sc, g, layers[i].flags & SMALL_MATH_MASK, aligned(layers[i].dst));
    }
};

struct Step {
    int form, layers;            // SMALL_FORM_*, layers covered
    Geom a, b;                   // of a pair in FP32, or a shortcut and the layer it joins
    int widths[13];              // of a chain of full reductions
    int fused;                   // of a fused pair (see fused_pair)
};

static void step_at(small_ctx *ctx, const small_layer *layers, int n_layers, int i, int N, const Forms &f, Step &s) {
    s.layers = 2;
    if (i == f.chain) { s.form = SMALL_FORM_PAIR_RUN; s.layers = f.chain_layers; return; }
    if (i == f.on_chip) { s.form = SMALL_FORM_ON_CHIP; s.layers = n_layers - i; return; }
    s.form = SMALL_FORM_PAIR_FP32;
    if (f.runs && f.chain < 0 && f.on_chip < 0 && split_pair(ctx, layers, n_layers, i, N, s.a, s.b) > 0.0) return;
    s.form = SMALL_FORM_JOINED;
    if (f.joins(ctx, layers, n_layers, i, N, s.a, s.b)) return;
    s.form = SMALL_FORM_FC_CHAIN;
    if (const int L = f.apart ? fc_chain_len(ctx, layers, n_layers, i, N, s.widths) : 0)
        if (f.aligned(layers[i + L - 1].dst)) { s.layers = L; return; }
    s.form = SMALL_FORM_FUSED_PAIR;
    if ((s.fused = i + 1 == f.on_chip || i + 1 == f.chain ? 0 : fused_pair(ctx, layers, n_layers, i, N))) return;
    // Two neighbouring layers that touch no common tensor except as readers (a residual stage's convolution and its
    // shortcut) run side by side.
    s.form = SMALL_FORM_SIDE_BY_SIDE;
    Geom sc, g;
    if (f.apart && ctx->branch_overlap && ctx->side_stream && i + 1 < n_layers && i + 1 != f.on_chip && i + 1 != f.chain && independent(layers[i], layers[i + 1]) &&
        !fused_pair(ctx, layers, n_layers, i + 1, N) && !f.joins(ctx, layers, n_layers, i + 1, N, sc, g))
        return;
    s.form = SMALL_FORM_LAYER;
    s.layers = 1;
}

}  // namespace small

using namespace small;

SMALL_API int small_set_net_fusion(small_ctx *ctx, unsigned mask) {
    if (!ctx) return SMALL_ERR_NOT_INIT;
    if (mask & ~(unsigned)(SMALL_FUSE_DWPW | SMALL_FUSE_DWPW_ALWAYS | SMALL_FUSE_CONVPOOL | SMALL_FUSE_FC_CHAIN | SMALL_FUSE_POOLFC)) return SMALL_ERR_INVALID_ARG;
    ctx->net_fusion = mask;
    return SMALL_OK;
}

SMALL_API int small_net_launches(small_ctx *ctx, const small_layer *layers, int n_layers, int N) {
    if (!ctx || !layers || n_layers < 1 || N < 1) return -1;
    int launches = 0;
    for (int i = 0; i < n_layers; ++i, ++launches) {
        int widths[13];
        if (const int L = fc_chain_len(ctx, layers, n_layers, i, N, widths)) i += L - 1;
        else if (fused_pair(ctx, layers, n_layers, i, N)) ++i;
    }
    return launches;
}

SMALL_API int small_net_forms(small_ctx *ctx, const small_layer *layers, int n_layers, int N, int *forms) {
    SlotPlan plan;
    if (!ctx || !plan_slots(layers, n_layers, N, plan)) return -1;
    const Forms f(ctx, layers, n_layers, 0, N, true, true);
    int launches = 0;
    Step step;
    for (int i = 0; i < n_layers; i += step.layers) {
        step_at(ctx, layers, n_layers, i, N, f, step);
        launches += step.form == SMALL_FORM_SIDE_BY_SIDE ? 2 : 1;
        for (int j = i; forms && j < i + step.layers; ++j) forms[j] = step.form;
    }
    return launches;
}

SMALL_API size_t small_net_workspace_bytes(const small_layer *layers, int n_layers, int N) {
    SlotPlan plan;
    if (!plan_slots(layers, n_layers, N, plan)) return 0;
    return plan.total;
}

static int run_layers(small_ctx *ctx, const small_layer *layers, int n_layers, int from, int N,
                      const float *in_blk, float *out_blk, void *workspace, size_t workspace_bytes, void *stream);

SMALL_API int small_run_net(small_ctx *ctx, const small_layer *layers, int n_layers, int N,
                            const float *in_blk, float *out_blk, void *workspace, size_t workspace_bytes, void *stream) {
    return run_layers(ctx, layers, n_layers, 0, N, in_blk, out_blk, workspace, workspace_bytes, stream);
}

// Validates the whole list, then runs layers from .. n_layers - 1.
static int run_layers(small_ctx *ctx, const small_layer *layers, int n_layers, int from, int N,
                      const float *in_blk, float *out_blk, void *workspace, size_t workspace_bytes, void *stream) {
    if (!ctx) return SMALL_ERR_NOT_INIT;
    if (!layers || !in_blk || !out_blk) return SMALL_ERR_INVALID_ARG;
    if (!aligned16(in_blk) || !aligned16(out_blk) || (workspace && ((uintptr_t)workspace & 255u))) return SMALL_ERR_ALIGN;
    SlotPlan plan;
    if (!plan_slots(layers, n_layers, N, plan)) return SMALL_ERR_SHAPE;
    if (plan.total > workspace_bytes || (plan.total && !workspace)) return SMALL_ERR_WORKSPACE;
    char *base = static_cast<char *>(workspace);
    auto rd = [&](int slot) -> const float * {
        if (slot == SMALL_SLOT_INPUT) return in_blk;
        if (slot == SMALL_SLOT_OUTPUT) return out_blk;
        return reinterpret_cast<const float *>(base + plan.offset[slot]);
    };
    auto wr = [&](int slot) -> float * {
        if (slot == SMALL_SLOT_OUTPUT) return out_blk;
        return reinterpret_cast<float *>(base + plan.offset[slot]);
    };
    // validate every layer before the first launch: weights present where needed, flags known
    for (int i = 0; i < n_layers; ++i) {
        const small_layer &L = layers[i];
        bool weighted = L.op == SMALL_OP_CONV || L.op == SMALL_OP_DWCONV || L.op == SMALL_OP_FC || L.op == SMALL_OP_DWPW || L.op == SMALL_OP_CONVPOOL;
        if (L.op == SMALL_OP_CONVPOOL &&
            !small_conv_maxpool_fused(N, L.C, L.K, L.H, L.W, L.FH, L.FW, L.stride, L.pad_t, L.pad_b, L.pad_l, L.pad_r))
            return SMALL_ERR_UNSUPPORTED;         // a network has no scratch tensor for the unfused form
        if (L.op == SMALL_OP_DWPW) {
            if (!L.w_blk2 || !aligned16(L.w_blk2) || (L.bias2 && !aligned16(L.bias2))) return SMALL_ERR_INVALID_ARG;
            if (!small_dwpw_fused(N, L.C, L.K, L.H, L.W, L.stride, L.pad_t, L.pad_b, L.pad_l, L.pad_r, L.flags & SMALL_MATH_MASK))
                return SMALL_ERR_UNSUPPORTED;     // a network has no scratch tensor for the unfused form
        }
        if (weighted && !L.w_blk) return SMALL_ERR_INVALID_ARG;
        if (weighted && (!aligned16(L.w_blk) || (L.bias && !aligned16(L.bias)))) return SMALL_ERR_ALIGN;
        unsigned allowed = L.op == SMALL_OP_CONV ? (SMALL_RELU | SMALL_ACCUMULATE | SMALL_MATH_MASK)
                         : (L.op == SMALL_OP_DWCONV || L.op == SMALL_OP_FC) ? (SMALL_RELU | SMALL_MATH_MASK)
                         : L.op == SMALL_OP_DWPW ? (SMALL_RELU | SMALL_RELU_MID | SMALL_MATH_MASK)
                         : L.op == SMALL_OP_CONVPOOL ? (SMALL_RELU | SMALL_MATH_MASK)
                         : L.op == SMALL_OP_ADD ? SMALL_RELU : 0u;
        if (L.flags & ~allowed) return SMALL_ERR_INVALID_ARG;
        if ((L.flags & SMALL_MATH_MASK) == SMALL_MATH_MASK) return SMALL_ERR_INVALID_ARG;
        if (L.op == SMALL_OP_POOL && L.pool_mode != SMALL_POOL_MAX && L.pool_mode != SMALL_POOL_AVG) return SMALL_ERR_INVALID_ARG;
        if (L.src == L.dst && L.op != SMALL_OP_RELU && L.op != SMALL_OP_ADD) return SMALL_ERR_OVERLAP;
    }
    auto run_one = [&](const small_layer &L, void *strm) -> int {
        switch (L.op) {
            case SMALL_OP_CONV:
                return small_conv2d(ctx, rd(L.src), L.w_blk, L.bias, wr(L.dst), N, L.C, L.K, L.H, L.W, L.FH, L.FW, L.stride,
                                 L.pad_t, L.pad_b, L.pad_l, L.pad_r, L.flags, strm);
            case SMALL_OP_DWCONV:
                return small_dwconv2d(ctx, rd(L.src), L.w_blk, L.bias, wr(L.dst), N, L.C, L.H, L.W, L.FH, L.FW, L.stride,
                                   L.pad_t, L.pad_b, L.pad_l, L.pad_r, L.flags, strm);
            case SMALL_OP_POOL:
                return small_pool2d(ctx, rd(L.src), wr(L.dst), nullptr, N, L.C, L.H, L.W, L.FH, L.FW, L.stride,
                                 L.pad_t, L.pad_b, L.pad_l, L.pad_r, L.pool_mode, strm);
            case SMALL_OP_RELU:
                return small_relu(ctx, rd(L.src), wr(L.dst), N, L.C, L.H, L.W, strm);
            case SMALL_OP_ADD:
                return small_add(ctx, rd(L.src), rd(L.src2), wr(L.dst), N, L.C, L.H, L.W, L.flags, strm);
            case SMALL_OP_FC:
                return small_fc(ctx, rd(L.src), L.w_blk, L.bias, wr(L.dst), N, L.C, L.K, L.flags, strm);
            case SMALL_OP_CONVPOOL:
                return small_conv_maxpool2d(ctx, rd(L.src), L.w_blk, L.bias, wr(L.dst), nullptr, N, L.C, L.K, L.H, L.W, L.FH, L.FW, L.stride,
                                         L.pad_t, L.pad_b, L.pad_l, L.pad_r, L.flags, strm);
            case SMALL_OP_DWPW:
                return small_dwpw_conv2d(ctx, rd(L.src), L.w_blk, L.bias, L.w_blk2, L.bias2, wr(L.dst), nullptr, N, L.C, L.K, L.H, L.W,
                                      L.stride, L.pad_t, L.pad_b, L.pad_l, L.pad_r, L.flags, strm);
        }
        return SMALL_ERR_INVALID_ARG;
    };
    struct InNet {
        small_ctx *ctx;
        ~InNet() { ctx->in_net = 0; ctx->dependent = 0; }
    } in_net{ctx};
    ctx->in_net = 1;
    bool after_join = false;
    const Forms forms(ctx, layers, n_layers, from, N, tensors_apart(plan, in_blk, out_blk, workspace), (reinterpret_cast<uintptr_t>(out_blk) & 31u) == 0);
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    Step step;
    for (int i = from; i < n_layers; i += step.layers) {
        const small_layer &L = layers[i];
        int s = SMALL_OK;
        // every layer may start its set-up while the kernel in front of it drains (see launch_kernel)
        ctx->dependent = !ctx->overlap || after_join ? 0 : i > 0 ? 1 : 2;
        after_join = false;
        step_at(ctx, layers, n_layers, i, N, forms, step);
        const small_layer &Nx = layers[i + step.layers - 1];      // the last one covered
        switch (step.form) {
            case SMALL_FORM_PAIR_RUN:
                s = launch_sep_chain(ctx, layers, n_layers, i, N, rd(L.src), wr(Nx.dst), st);
                break;
            case SMALL_FORM_ON_CHIP:
                s = launch_resident(ctx, layers, n_layers, from, N, rd, wr, st);
                break;
            case SMALL_FORM_PAIR_FP32:
                s = launch_split_pair(ctx, rd(L.src), L.w_blk, L.bias, L.flags & SMALL_RELU, Nx.w_blk, Nx.bias, wr(Nx.dst), step.a, step.b, Nx.flags & SMALL_RELU, st);
                break;
            case SMALL_FORM_JOINED:
                s = launch_joined(ctx, Shortcut{rd(L.src), L.w_blk, nullptr, nullptr, L.bias, step.a}, rd(Nx.src), Nx.w_blk, Nx.bias, wr(L.dst), step.b, Nx.flags & SMALL_RELU,
                                  L.flags & SMALL_MATH_MASK, st);
                break;
            case SMALL_FORM_FC_CHAIN: {
                const float *w[12], *b[12];
                int relu[12];
                for (int j = 0; j < step.layers; ++j) { w[j] = layers[i + j].w_blk; b[j] = layers[i + j].bias; relu[j] = (layers[i + j].flags & SMALL_RELU) ? 1 : 0; }
                s = launch_fc_chain(ctx, rd(L.src), w, b, step.widths, relu, wr(Nx.dst), step.layers, N, L.flags & SMALL_MATH_MASK, st);
                break;
            }
            case SMALL_FORM_FUSED_PAIR:
                if (step.fused == SMALL_OP_DWPW) {
                    const unsigned fl = ((L.flags & SMALL_RELU) ? SMALL_RELU_MID : 0u) | (Nx.flags & (SMALL_RELU | SMALL_MATH_MASK));
                    s = small_dwpw_conv2d(ctx, rd(L.src), L.w_blk, L.bias, Nx.w_blk, Nx.bias, wr(Nx.dst), nullptr, N, L.C, Nx.K, L.H, L.W,
                                          L.stride, L.pad_t, L.pad_b, L.pad_l, L.pad_r, fl, stream);
                } else if (step.fused == kFusedPoolFc) {
                    s = small_gap_fc(ctx, rd(L.src), Nx.w_blk, Nx.bias, wr(Nx.dst), nullptr, N, L.C, L.H, L.W, Nx.K,
                                     Nx.flags & (SMALL_RELU | SMALL_MATH_MASK), stream);
                } else {
                    s = small_conv_maxpool2d(ctx, rd(L.src), L.w_blk, L.bias, wr(Nx.dst), nullptr, N, L.C, L.K, L.H, L.W, L.FH, L.FW, L.stride,
                                             L.pad_t, L.pad_b, L.pad_l, L.pad_r, L.flags, stream);
                }
                break;
            case SMALL_FORM_SIDE_BY_SIDE: {
                // the second one on the context's side stream, forked from and joined to the caller's stream by events, so that a
                // short layer hides behind a long one.  It is an ordinary launch, and so is the layer behind the join.
                cudaStream_t side = static_cast<cudaStream_t>(ctx->side_stream);
                cudaError_t e = cudaEventRecord(static_cast<cudaEvent_t>(ctx->ev_fork), st);
                if (e == cudaSuccess) e = cudaStreamWaitEvent(side, static_cast<cudaEvent_t>(ctx->ev_fork), 0);
                if (e != cudaSuccess) { ctx->last_cuda = (int)e; ctx->dependent = 0; return SMALL_ERR_CUDA; }
                s = run_one(L, stream);
                ctx->dependent = 0;
                if (s == SMALL_OK) s = run_one(Nx, ctx->side_stream);
                e = cudaEventRecord(static_cast<cudaEvent_t>(ctx->ev_join), side);
                if (e == cudaSuccess) e = cudaStreamWaitEvent(st, static_cast<cudaEvent_t>(ctx->ev_join), 0);
                if (s == SMALL_OK && e != cudaSuccess) { ctx->last_cuda = (int)e; s = SMALL_ERR_CUDA; }
                after_join = true;
                break;
            }
            default:
                s = run_one(L, stream);
        }
        ctx->dependent = 0;
        if (s != SMALL_OK) return s;
    }
    return SMALL_OK;
}

SMALL_API size_t small_net_host_staging_bytes(int N, int C, int H, int W, int outC, int outH, int outW) {
    if (N < 1 || C < 1 || H < 1 || W < 1 || outC < 1 || outH < 1 || outW < 1) return 0;
    return 2 * round256(sizeof(float) * (size_t)N * C * H * W) + round256(sizeof(float) * packed_elems(N, C, H, W)) +
           round256(sizeof(float) * packed_elems(N, outC, outH, outW)) + round256(sizeof(float) * (size_t)N * outC * outH * outW);
}

// The staging areas of a workspace: the entry of the calls before on the same memory, laid out alike, or a new one (`fresh`),
// which takes the place of every entry whose memory it overlaps, or of the one unused for longest.
static small_host_stage &host_stage(small_ctx *ctx, const char *base, size_t bytes, const char *in, size_t in_bytes, bool &fresh) {
    const unsigned long long now = ++ctx->host_calls;
    for (small_host_stage &h : ctx->host_stage)
        if (h.base == base && h.bytes == bytes && h.in == in && h.in_bytes == in_bytes) { fresh = false; h.last = now; return h; }
    int ordered = 0;
    small_host_stage *pick = nullptr;
    auto rank = [](const small_host_stage &h) { return h.base ? (h.ordered ? 2 : 1) : 0; };
    for (small_host_stage &h : ctx->host_stage) {
        if (h.base && base < h.base + h.bytes && h.base < base + bytes) { ordered |= h.ordered; h.base = nullptr; }
        if (!pick || rank(h) < rank(*pick) || (rank(h) == rank(*pick) && h.last < pick->last)) pick = &h;
    }
    if (rank(*pick) == 2) ctx->host_ordered = 1;
    pick->base = base; pick->bytes = bytes; pick->in = in; pick->in_bytes = in_bytes;
    pick->next = pick->used[0] = pick->used[1] = 0; pick->ordered = ordered; pick->last = now;
    fresh = true;
    return *pick;
}

// The host-buffer call keeps the copy engine busy next to the SMs: the NCHW input goes to one of two staging areas on
// the context's copy stream, so the copy of call i + 1 runs while the layers of call i are still computing on the caller's
// stream; the caller's stream waits for its own input by an event, and a staging area is not overwritten before the
// layer that read it last has finished.  The first copy into a workspace waits for everything in front of it on the caller's
// stream, which may still use that memory for something else, and so does every copy once a call was captured on it.  Everything else (pack, layers, unpack, the result's copy back)
// stays in order on the caller's stream.  While the caller's stream is being captured, the input copy stays on that stream.
SMALL_API int small_run_net_host(small_ctx *ctx, const small_layer *layers, int n_layers, int N,
                                 const float *in_host, int C, int H, int W,
                                 float *out_host, int outC, int outH, int outW,
                                 void *workspace, size_t workspace_bytes, void *stream) {
    if (!ctx) return SMALL_ERR_NOT_INIT;
    if (!layers || !in_host || !out_host || !workspace) return SMALL_ERR_INVALID_ARG;
    if ((uintptr_t)workspace & 255u) return SMALL_ERR_ALIGN;
    {   // the layer list must be well formed even when it needs no slot
        SlotPlan plan;
        if (!plan_slots(layers, n_layers, N, plan)) return SMALL_ERR_SHAPE;
    }
    size_t net_b = small_net_workspace_bytes(layers, n_layers, N);
    size_t stage_b = small_net_host_staging_bytes(N, C, H, W, outC, outH, outW);
    if (stage_b == 0) return SMALL_ERR_SHAPE;
    if (net_b + stage_b > workspace_bytes) return SMALL_ERR_WORKSPACE;
    // the last layer must produce the declared output shape
    int oc, oh, ow;
    if (!layer_out_shape(layers[n_layers - 1], N, oc, oh, ow) || oc != outC || oh != outH || ow != outW) return SMALL_ERR_SHAPE;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    char *p = static_cast<char *>(workspace) + net_b;
    size_t in_nchw_b = sizeof(float) * (size_t)N * C * H * W, out_nchw_b = sizeof(float) * (size_t)N * outC * outH * outW;
    float *d_in_nchw[2];
    d_in_nchw[0] = reinterpret_cast<float *>(p); p += round256(in_nchw_b);
    d_in_nchw[1] = reinterpret_cast<float *>(p); p += round256(in_nchw_b);
    float *d_in_blk = reinterpret_cast<float *>(p); p += round256(sizeof(float) * packed_elems(N, C, H, W));
    float *d_out_blk = reinterpret_cast<float *>(p); p += round256(sizeof(float) * packed_elems(N, outC, outH, outW));
    float *d_out_nchw = reinterpret_cast<float *>(p);
    cudaError_t e = cudaSuccess;
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    cudaStreamIsCapturing(st, &cap);
    const bool piped = ctx->copy_stream && cap == cudaStreamCaptureStatusNone;
    int par = 0;
    bool fresh = true;
    small_host_stage *stage = nullptr;
    if (ctx->copy_stream) {
        stage = &host_stage(ctx, static_cast<const char *>(workspace), net_b + stage_b, reinterpret_cast<const char *>(d_in_nchw[0]), in_nchw_b, fresh);
        if (!piped) stage->ordered = 1;
        if (stage->ordered || ctx->host_ordered) fresh = true;
    }
    if (piped) {
        par = stage->next;
        cudaStream_t cs = static_cast<cudaStream_t>(ctx->copy_stream);
        if (fresh) {           // behind everything queued so far
            e = cudaEventRecord(static_cast<cudaEvent_t>(ctx->ev_start), st);
            if (e == cudaSuccess) e = cudaStreamWaitEvent(cs, static_cast<cudaEvent_t>(ctx->ev_start), 0);
        } else if (stage->used[par]) {
            e = cudaStreamWaitEvent(cs, static_cast<cudaEvent_t>(stage->ev_read[par]), 0);
        }
        if (e == cudaSuccess) e = cudaMemcpyAsync(d_in_nchw[par], in_host, in_nchw_b, cudaMemcpyHostToDevice, cs);
        if (e == cudaSuccess) e = cudaEventRecord(static_cast<cudaEvent_t>(ctx->ev_h2d), cs);
        if (e == cudaSuccess) e = cudaStreamWaitEvent(st, static_cast<cudaEvent_t>(ctx->ev_h2d), 0);
    } else {
        e = cudaMemcpyAsync(d_in_nchw[0], in_host, in_nchw_b, cudaMemcpyHostToDevice, st);
    }
    if (e != cudaSuccess) {
        if (stage && !stage->ordered) stage->base = nullptr;
        ctx->last_cuda = (int)e;
        return SMALL_ERR_CUDA;
    }
    // A first layer with at most four input channels (an image, a spectrogram) reads the NCHW tensor itself: its kernel
    // gathers the real channels into shared memory either way, so the blocked copy of the input - 32 lanes for one to four
    // channels - is never made.  The values and their order of summation are those of the blocked path.
    int first = 0;
    {
        const small_layer &L0 = layers[0];
        Geom g0;
        bool later_reads_input = false;
        for (int i = 1; i < n_layers; ++i)
            if (layers[i].src == SMALL_SLOT_INPUT || (layers[i].op == SMALL_OP_ADD && layers[i].src2 == SMALL_SLOT_INPUT)) later_reads_input = true;
        if (L0.op == SMALL_OP_CONV && L0.src == SMALL_SLOT_INPUT && L0.dst >= 0 && !(L0.flags & SMALL_ACCUMULATE) && !later_reads_input &&
            n_layers > 1 && L0.C == C && L0.H == H && L0.W == W && L0.w_blk && aligned16(L0.w_blk) && (!L0.bias || aligned16(L0.bias)) &&
            !(L0.flags & ~(SMALL_RELU | SMALL_MATH_MASK)) && !fused_pair(ctx, layers, n_layers, 0, N) &&
            make_geom(g0, N, L0.C, L0.K, L0.H, L0.W, L0.FH, L0.FW, L0.stride, L0.pad_t, L0.pad_b, L0.pad_l, L0.pad_r) == SMALL_OK &&
            conv_thin_supported(g0)) {
            SlotPlan plan;
            plan_slots(layers, n_layers, N, plan);
            float *dst0 = reinterpret_cast<float *>(static_cast<char *>(workspace) + plan.offset[L0.dst]);
            if (int s = launch_conv_thin(ctx, d_in_nchw[par], L0.w_blk, L0.bias, dst0, g0, L0.flags & SMALL_RELU, false, st, true)) return s;
            first = 1;
        }
    }
    if (!first)
        if (int s = small_pack(ctx, d_in_nchw[par], d_in_blk, N, C, H, W, stream)) return s;
    if (piped) {
        e = cudaEventRecord(static_cast<cudaEvent_t>(stage->ev_read[par]), st);
        if (e != cudaSuccess) { ctx->last_cuda = (int)e; return SMALL_ERR_CUDA; }
        stage->used[par] = 1;
        stage->next = par ^ 1;
    }
    if (first) {
        // the rest of the list over the same slots: its plan must be the whole list's (slot sizes come from all layers)
        if (int s = run_layers(ctx, layers, n_layers, 1, N, d_in_blk, d_out_blk, workspace, net_b, stream)) return s;
    } else if (int s = small_run_net(ctx, layers, n_layers, N, d_in_blk, d_out_blk, workspace, net_b, stream)) return s;
    if (int s = small_unpack(ctx, d_out_blk, d_out_nchw, N, outC, outH, outW, stream)) return s;
    e = cudaMemcpyAsync(out_host, d_out_nchw, out_nchw_b, cudaMemcpyDeviceToHost, st);
    if (e != cudaSuccess) { ctx->last_cuda = (int)e; return SMALL_ERR_CUDA; }
    return SMALL_OK;
}
