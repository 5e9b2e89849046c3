"""The work that users of this library have it do, as cases to time.

Three kinds of pass:

  net     one of the four networks of synth/configs.py through the network runner: `Net.run` on a batch that is resident
          in device memory in the blocked layout, or `Net.run_host` from pinned host memory to pinned host memory.
          Batches from a single image (what the paper measures on its boards) up to each network's own full batch.
  layer   one float layer called on its own (`small_conv2d`, `small_dwconv2d`, `small_pool2d`), as a program does that
          runs its own model layer by layer: the layer sweep of the benchmark and ragged shapes like it.
  quant   uint8 layers (`small_q_*`): a convolution, or a depthwise-separable block followed by max pooling.

Float convolutions and full reductions run in one of the three math modes (fp32, tf32, 3xtf32), which the caller picks.
"""
import math

import torch

from paper_2303_04769_b200 import binding as B
from paper_2303_04769_b200.net import Net
from synth import configs

FULL_BATCH = {"residual_cnn": 256, "dwsep_cnn": 64, "kws_cnn": 1024, "autoencoder_fc": 4096}


def _net(name, net, batch, mode, entry="device"):
    return dict(name=name, kind="net", net=net, batch=batch, math=mode, entry=entry)


def _conv(name, mode, N, C, K, H, W, F, S):
    return dict(name=name, kind="layer", op="conv", math=mode, N=N, C=C, K=K, H=H, W=W, F=F, S=S)


def listed():
    return [
        # one image at a time: the paper's end-to-end latency (Section 5.4), where launches and host work count
        _net("residual_b1_3xtf32", "residual_cnn", 1, "3xtf32"),
        # the benchmark's step: offline inference on a full batch at FP32 accuracy
        _net("residual_b256_3xtf32", "residual_cnn", 256, "3xtf32"),
        # the deepest network, 29 layers that shrink to 3 x 3 planes
        _net("dwsep_b64_3xtf32", "dwsep_cnn", 64, "3xtf32"),
        # serving from host buffers: copy in, network, copy out
        _net("kws_b1024_3xtf32_host", "kws_cnn", 1024, "3xtf32", "host"),
        # a small odd batch in the default math mode of `Net`
        _net("kws_b37_fp32", "kws_cnn", 37, "fp32"),
        # full reductions only, large batch, the fastest math mode
        _net("autoencoder_b4096_tf32", "autoencoder_fc", 4096, "tf32"),
        # the layer sweep: the largest 3x3 plane in the accurate tensor-core mode, a 3x3 in FP32, a depthwise layer
        _conv("conv3x3_c64_hw56_3xtf32", "3xtf32", 128, 64, 64, 56, 56, 3, 1),
        _conv("conv3x3_c256_hw14_fp32", "fp32", 128, 256, 256, 14, 14, 3, 1),
        # a pointwise layer whose channels, filters and plane are no round numbers
        _conv("conv1x1_ragged_tf32", "tf32", 50, 200, 136, 31, 29, 1, 1),
        dict(name="dw3x3_c64_hw56", kind="layer", op="dw", N=128, C=64, H=56, W=56, S=1),
        # quantised models (Section 5.1): a residual network's inner layer, and a depthwise-separable block with pooling
        dict(name="qconv3x3_c64_hw28", kind="quant", op="conv", N=128, C=64, K=64, H=28, W=28, F=3, S=1),
        dict(name="qblock_c64_hw25x5", kind="quant", op="block", N=512, C=64, K=64, H=25, W=5, S=1),
    ]


def _log(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi + 0.49)))))))


def draw(rng):
    kind = rng.choice(["net", "net", "net", "net", "layer", "layer", "layer", "quant"])
    if kind == "net":
        net = rng.choice(sorted(FULL_BATCH))
        return dict(kind="net", net=net, batch=_log(rng, 1, FULL_BATCH[net]), math=rng.choice(["fp32", "tf32", "3xtf32"]),
                    entry=rng.choice(["device", "device", "host"]))
    H = _log(rng, 5, 56)
    W = max(4, min(56, H + rng.randint(-3, 3)))
    N, S = _log(rng, 1, 128), rng.choice([1, 1, 1, 2])
    if kind == "layer":
        op = rng.choice(["conv", "conv", "conv", "dw", "pool"])
        if op != "conv":
            case = dict(kind="layer", op=op, N=N, C=_log(rng, 8, 512), H=H, W=W, S=2 if op == "pool" else S)
            if op == "pool":
                case["F"] = rng.choice([2, 3])
        else:
            case = dict(kind="layer", op="conv", math=rng.choice(["fp32", "tf32", "3xtf32"]), N=N, C=_log(rng, 8, 512),
                        K=_log(rng, 8, 512), H=H, W=W, F=rng.choice([1, 3]), S=S)
    elif rng.random() < 0.6:
        case = dict(kind="quant", op="conv", N=N, C=_log(rng, 8, 256), K=_log(rng, 8, 256), H=H, W=W, F=rng.choice([1, 3]), S=S)
    else:
        case = dict(kind="quant", op="block", N=N, C=_log(rng, 8, 256), K=_log(rng, 8, 256), H=H, W=W, S=S)
    # no drawn layer is larger than the largest listed one: smaller batches for wide layers on large planes
    pointwise = case["op"] == "block" or case.get("F") == 1
    most = {"fp32": 12e9, "tf32": 29e9, "3xtf32": 29e9}.get(case.get("math"), 12e9) / (4 if pointwise else 1)
    while case["N"] > 1 and (work(case)["flops"] > most or work(case)["bytes"] > 206e6):
        case["N"] = (case["N"] + 1) // 2
    return case


# ---- prepare


def _ctx():
    device = torch.cuda.current_device()
    if device not in _ctx.made:
        _ctx.made[device] = B.small_init(device)
    return _ctx.made[device]


_ctx.made = {}


def _rand(gen, shape, lo, hi):
    return torch.rand(shape, generator=gen, device="cuda") * (hi - lo) + lo


def _blocked(ctx, nchw):
    N, C, H, W = nchw.shape
    blk = torch.empty(B.small_packed_elems(N, C, H, W), device="cuda")
    B.small_pack(ctx, nchw, blk, N, C, H, W)
    return blk


def _bytes(gen, shape, mean, std):
    return (torch.randn(shape, generator=gen, device="cuda") * std + mean).round().clamp(0, 255).to(torch.uint8)


def _q_blocked(ctx, nchw):
    N, C, H, W = nchw.shape
    blk = torch.empty(B.small_q_packed_bytes(N, C, H, W), dtype=torch.uint8, device="cuda")
    B.small_q_pack(ctx, nchw, blk, N, C, H, W)
    return blk


def _q_params(terms):
    """Zero points and the fixed-point scale of a quantised layer of `terms` products: results spread over the byte range."""
    return (6, 128, 9, int(40.0 / (60.0 * 30.0 * math.sqrt(terms)) * 2 ** 36), 36)


def prepare(case, seed):
    ctx, gen = _ctx(), torch.Generator(device="cuda").manual_seed(seed)
    state = dict(case=case, ctx=ctx)
    if case["kind"] == "net":
        desc = configs.NETWORKS[case["net"]](case["batch"])
        shape = (case["batch"],) + tuple(desc["input"])
        kind, a, b = desc["input_dist"]
        x = _rand(gen, shape, a, b) if kind == "uniform" else torch.randn(shape, generator=gen, device="cuda") * b + a
        state["net"] = Net(ctx, desc, configs.make_params(desc, seed), math=case["math"])
        if case["entry"] == "host":
            state["in"] = x.cpu().pin_memory()
            state["out"] = torch.empty((case["batch"],) + tuple(state["net"].out_shape)).pin_memory()
        else:
            state["in"] = _blocked(ctx, x)
        return state
    N, C, H, W, S, F = case["N"], case["C"], case["H"], case["W"], case["S"], case.get("F", 3)
    p = 1 if F == 3 else 0
    OH, OW = B.small_out_size(H, F, S, p, p), B.small_out_size(W, F, S, p, p)
    state.update(F=F, pad=(p, p, p, p))
    if case["kind"] == "layer":
        state["in"] = _blocked(ctx, _rand(gen, (N, C, H, W), -1.0, 1.0))
        K = case.get("K", C)
        state["out"] = torch.empty(B.small_packed_elems(N, K, OH, OW), device="cuda")
        if case["op"] == "conv":
            mode = B.MATH[case["math"]]
            state["w"] = torch.empty(B.small_conv_weight_elems(C, K, F, F, mode), device="cuda")
            B.small_pack_conv_weights(ctx, _rand(gen, (K, C, F, F), -1.0, 1.0), state["w"], C, K, F, F, mode)
        elif case["op"] == "dw":
            state["w"] = torch.empty(B.small_dw_weight_elems(C, 3, 3), device="cuda")
            B.small_pack_dw_weights(ctx, _rand(gen, (C, 3, 3), -1.0, 1.0), state["w"], C, 3, 3)
        state["bias"] = _rand(gen, (K,), -1.0, 1.0)
        return state
    # quantised: activations behind a ReLU (zero point near 0), filters around the middle of the byte range
    state["in"] = _q_blocked(ctx, _bytes(gen, (N, C, H, W), 6, 60))
    K = case["K"]
    state["out"] = torch.empty(B.small_q_packed_bytes(N, K, OH, OW), dtype=torch.uint8, device="cuda")
    FP = F if case["op"] == "conv" else 1
    state["w"] = torch.empty(B.small_q_conv_weight_bytes(C, K, FP, FP), dtype=torch.uint8, device="cuda")
    B.small_q_pack_conv_weights(ctx, _bytes(gen, (K, C, FP, FP), 128, 30), state["w"], C, K, FP, FP)
    state["bias"] = torch.randint(-2000, 2001, (K,), generator=gen, device="cuda", dtype=torch.int32)
    state["qp"] = _q_params(C * FP * FP)
    if case["op"] == "block":
        state["dw"] = torch.empty(B.small_q_dw_weight_bytes(C, 3, 3), dtype=torch.uint8, device="cuda")
        B.small_q_pack_dw_weights(ctx, _bytes(gen, (C, 3, 3), 128, 30), state["dw"], C, 3, 3)
        state["dw_bias"] = torch.randint(-2000, 2001, (C,), generator=gen, device="cuda", dtype=torch.int32)
        state["dw_qp"] = _q_params(9)
        state["mid"] = torch.empty(B.small_q_packed_bytes(N, C, OH, OW), dtype=torch.uint8, device="cuda")
        state["pooled"] = torch.empty(B.small_q_packed_bytes(N, K, OH // 2, OW // 2), dtype=torch.uint8, device="cuda")
    return state


# ---- run


def run(state):
    case, ctx = state["case"], state["ctx"]
    if case["kind"] == "net":
        if case["entry"] == "host":
            state["net"].run_host(state["in"], state["out"])
            return state["out"]
        return state["net"].run(state["in"])
    N, C, H, W, S, F, pad, out = case["N"], case["C"], case["H"], case["W"], case["S"], state["F"], state["pad"], state["out"]
    if case["kind"] == "layer":
        if case["op"] == "conv":
            B.small_conv2d(ctx, state["in"], state["w"], state["bias"], out, N, C, case["K"], H, W, F, F, S, pad, B.RELU | B.MATH[case["math"]])
        elif case["op"] == "dw":
            B.small_dwconv2d(ctx, state["in"], state["w"], state["bias"], out, N, C, H, W, 3, 3, S, pad, B.RELU)
        else:
            B.small_pool2d(ctx, state["in"], out, None, N, C, H, W, F, F, S, pad, B.POOL_MAX)
        return out
    if case["op"] == "conv":
        B.small_q_conv2d(ctx, state["in"], state["w"], state["bias"], out, N, C, case["K"], H, W, F, F, S, pad, state["qp"], B.RELU)
        return out
    OH, OW = B.small_out_size(H, 3, S, 1, 1), B.small_out_size(W, 3, S, 1, 1)
    B.small_q_dwconv2d(ctx, state["in"], state["dw"], state["dw_bias"], state["mid"], N, C, H, W, 3, 3, S, pad, state["dw_qp"], B.RELU)
    B.small_q_conv2d(ctx, state["mid"], state["w"], state["bias"], out, N, C, case["K"], OH, OW, 1, 1, 1, (0, 0, 0, 0), state["qp"], B.RELU)
    B.small_q_maxpool2d(ctx, out, state["pooled"], N, case["K"], OH, OW, 2, 2, 2, (0, 0, 0, 0), state["qp"][2])
    return out, state["pooled"]


# ---- what a pass needs at least, and how far two correct implementations may differ


def _out(I, F, S, pad):
    return (I + 2 * pad - F) // S + 1


def work(case):
    if case["kind"] == "net":
        desc, N = configs.NETWORKS[case["net"]](case["batch"]), case["batch"]
        dims, flops, params = {"in": tuple(desc["input"])}, 0, 0
        for L in desc["layers"]:
            _, h, w = dims[L["src"]]
            fh, fw = (L["FH"], L["FW"]) if L["FH"] else (h, w)
            pt, pb, pl, pr = L["pad"]
            oh, ow = (h + pt + pb - fh) // L["stride"] + 1, (w + pl + pr - fw) // L["stride"] + 1
            dims[L["dst"]] = (L["K"], oh, ow)
            taps = fh * fw * (L["C"] if L["op"] in ("conv", "fc") else 1)
            flops += (1 if L["op"] == "pool" else 2) * N * oh * ow * L["K"] * taps
            params += 0 if L["op"] == "pool" else L["K"] * (taps + 1)
        return {"bytes": 4.0 * (N * math.prod(dims["in"]) + N * math.prod(dims["out"]) + params), "flops": float(flops)}
    N, C, H, W, S, F = case["N"], case["C"], case["H"], case["W"], case["S"], case.get("F", 3)
    K, p = case.get("K", C), 1 if F == 3 else 0
    OH, OW = _out(H, F, S, p), _out(W, F, S, p)
    pixels = N * OH * OW
    if case["kind"] == "layer":
        moved = 4.0 * (N * C * H * W + pixels * K)
        if case["op"] == "conv":
            return {"bytes": moved + 4.0 * K * (C * F * F + 1), "flops": 2.0 * pixels * K * C * F * F}
        if case["op"] == "dw":
            return {"bytes": moved + 4.0 * 10 * C, "flops": 2.0 * pixels * C * 9}
        return {"bytes": moved, "flops": 1.0 * pixels * C * F * F}
    moved = 1.0 * (N * C * H * W + pixels * K)
    if case["op"] == "conv":
        return {"bytes": moved + K * (C * F * F + 4.0), "flops": 2.0 * pixels * K * C * F * F}
    return {"bytes": moved + N * K * (OH // 2) * (OW // 2) + K * (C + 4.0) + 13.0 * C, "flops": 2.0 * pixels * C * (9 + K)}


def tolerance(case):
    if case["kind"] == "quant" or case.get("op") == "pool":
        return "exact"                      # integer layers and maxima are exact by definition
    if case.get("op") == "dw" or case["math"] == "fp32":
        return {"rel": 1e-5}                # sums of 32-bit products
    deep = case.get("net") == "autoencoder_fc"     # ten full reductions in a row amplify each layer's rounding
    if case["math"] == "3xtf32":
        return {"rel": 3e-5 if deep else 1e-5}
    return {"rel": 7e-3 if deep else 3e-3}  # products of 11-bit significands
