"""Layers called on their own start their set-up while the kernel in front of them drains.  What they read - the tensor, the filters,
the bias - may have been written by exactly that kernel: nothing of it may be read before it is there."""
import pytest
import torch

from synth import configs
from paper_2303_04769_b200 import binding as B
from paper_2303_04769_b200.net import Net
from gpu_util import ctx, to_blk

pytestmark = pytest.mark.gpu
P1, P0 = (1, 1, 1, 1), (0, 0, 0, 0)

CONVS = [  # N, C, K, H, W, F, S, mode: one for every kernel family
    (64, 3, 16, 32, 32, 3, 1, "fp32"), (64, 16, 16, 32, 32, 3, 1, "3xtf32"), (32, 64, 64, 20, 20, 3, 1, "3xtf32"), (32, 64, 64, 20, 20, 1, 1, "tf32"),
    (16, 64, 64, 14, 14, 3, 1, "fp32"), (2, 40, 40, 6, 5, 3, 1, "fp32"), (16, 64, 300, 9, 9, 3, 2, "tf32"),
]


def make(case, i):
    N, C, K, H, W, F, S, mode = case
    g = torch.Generator(device="cuda").manual_seed(i)
    return (torch.rand(B.small_packed_elems(N, C, H, W), generator=g, device="cuda"), torch.rand((K, C, F, F), generator=g, device="cuda") - 0.5,
            torch.rand((K,), generator=g, device="cuda") - 0.5)


def conv(case, x, wb, b, out):
    N, C, K, H, W, F, S, mode = case
    B.small_conv2d(ctx(), x, wb, b, out, N, C, K, H, W, F, F, S, P1 if F == 3 else P0, B.RELU | B.MATH[mode])


@pytest.mark.parametrize("case", CONVS)
def test_filters_bias_and_input_written_just_before(case):
    N, C, K, H, W, F, S, mode = case
    p = 1 if F == 3 else 0
    OH, OW = B.small_out_size(H, F, S, p, p), B.small_out_size(W, F, S, p, p)
    sets = [make(case, i) for i in range(6)]
    wb = torch.empty(B.small_conv_weight_elems(C, K, F, F, B.MATH[mode]), device="cuda")
    new = lambda: torch.full((B.small_packed_elems(N, K, OH, OW),), float("nan"), device="cuda")
    want = []
    try:
        B.small_set_layer_overlap(ctx(), 0)
        for x, w, b in sets:
            B.small_pack_conv_weights(ctx(), w, wb, C, K, F, F, B.MATH[mode])
            want.append(new())
            conv(case, x, wb, b, want[-1])
            torch.cuda.synchronize()
    finally:
        B.small_set_layer_overlap(ctx(), 1)
    x_in, b_in, packed = torch.empty_like(sets[0][0]), torch.empty_like(sets[0][2]), [torch.empty_like(wb) for _ in sets]
    for (x, w, b), pw in zip(sets, packed):
        B.small_pack_conv_weights(ctx(), w, pw, C, K, F, F, B.MATH[mode])
    torch.cuda.synchronize()
    for trial in range(40):
        i = trial % len(sets)
        x, w, b = sets[i]
        out = new()
        order = trial % 4                         # what the kernel right in front of the layer writes: filters (two ways), bias, input
        steps = [lambda: x_in.copy_(x), lambda: b_in.copy_(b), lambda: B.small_pack_conv_weights(ctx(), w, wb, C, K, F, F, B.MATH[mode]),
                 lambda: torch.mul(packed[i], 1.0, out=wb)]
        for s in [s for j, s in enumerate(steps) if j != order and not (order == 3 and j == 2)] + [steps[order]]:
            s()
        conv(case, x_in, wb, b_in, out)
        conv(case, x_in, wb, b_in, out)           # and behind a layer of its own kind, over its output
        assert torch.equal(out, want[i]), (trial, order)
    assert B.small_device_status(ctx()) == 0


def test_chains_of_calls_keep_their_order():
    """Depthwise, 1x1, pooling and element-wise layers called one after the other on the same two tensors."""
    N, C, H = 48, 64, 24
    x0 = torch.rand(B.small_packed_elems(N, C, H, H), device="cuda") - 0.5
    dw, cw = torch.empty(B.small_dw_weight_elems(C, 3, 3), device="cuda"), torch.empty(B.small_conv_weight_elems(C, C, 1, 1, B.MATH_3XTF32), device="cuda")
    B.small_pack_dw_weights(ctx(), torch.rand((C, 3, 3), device="cuda") - 0.5, dw, C, 3, 3)
    B.small_pack_conv_weights(ctx(), (torch.rand((C, C, 1, 1), device="cuda") - 0.5) * 0.3, cw, C, C, 1, 1, B.MATH_3XTF32)

    def run():
        a, b, small = x0.clone(), torch.empty_like(x0), torch.empty(B.small_packed_elems(N, C, H // 2, H // 2), device="cuda")
        for _ in range(4):
            B.small_dwconv2d(ctx(), a, dw, None, b, N, C, H, H, 3, 3, 1, P1, B.RELU)
            B.small_conv2d(ctx(), b, cw, None, a, N, C, C, H, H, 1, 1, 1, P0, B.MATH_3XTF32)
            B.small_add(ctx(), a, x0, b, N, C, H, H, 0)
            B.small_relu(ctx(), b, a, N, C, H, H)
        B.small_pool2d(ctx(), a, small, None, N, C, H, H, 2, 2, 2, P0, B.POOL_MAX)
        return small

    try:
        B.small_set_layer_overlap(ctx(), 0)
        want = run()
        torch.cuda.synchronize()
    finally:
        B.small_set_layer_overlap(ctx(), 1)
    for _ in range(10):
        assert torch.equal(run(), want)


@pytest.mark.parametrize("name,batch", [("kws_cnn", 64), ("dwsep_cnn", 16), ("residual_cnn", 40), ("autoencoder_fc", 500)])
@pytest.mark.parametrize("math", ["fp32", "tf32"])
def test_network_right_behind_its_parameters(name, batch, math):
    """The first layer of a network is a dependent launch too: filters of any layer may come from the kernel in front of it."""
    net = configs.NETWORKS[name](batch=batch)
    nets = [Net(ctx(), net, configs.make_params(net, seed), batch=batch, math=math) for seed in range(3)]
    blk = to_blk(configs.make_input(net, batch))
    want = [n.run(blk).clone() for n in nets]
    weights = [[t for t in n.keep if isinstance(t, torch.Tensor)] for n in nets]
    torch.cuda.synchronize()
    for trial in range(24):
        i = 1 + trial % 2
        pairs = list(zip(weights[0], weights[i]))
        for dst, src in pairs[trial % len(pairs):] + pairs[:trial % len(pairs)]:      # another tensor is the last one each time
            torch.mul(src, 1, out=dst)
        assert torch.equal(nets[0].run(blk), want[i])


def test_capture_behind_copies_and_forks():
    case = CONVS[3]
    N, C, K, H, W, F, S, mode = case
    x, w, b = make(case, 1)
    wb = torch.empty(B.small_conv_weight_elems(C, K, F, F, B.MATH[mode]), device="cuda")
    B.small_pack_conv_weights(ctx(), w, wb, C, K, F, F, B.MATH[mode])
    want, out, x_in = (torch.empty(B.small_packed_elems(N, K, H, W), device="cuda"), torch.empty(B.small_packed_elems(N, K, H, W), device="cuda"), torch.empty_like(x))
    conv(case, x, wb, b, want)
    torch.cuda.synchronize()
    graph, side = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    with torch.cuda.graph(graph):
        x_in.copy_(x)                              # a copy node in front of the layer
        conv(case, x_in, wb, b, out)
        main = torch.cuda.current_stream()
        side.wait_stream(main)
        with torch.cuda.stream(side):
            x_in.zero_()
            x_in.add_(x)
        main.wait_stream(side)                     # and a join
        conv(case, x_in, wb, b, out)
    for _ in range(3):
        out.fill_(float("nan"))
        graph.replay()
        assert torch.equal(out, want)
