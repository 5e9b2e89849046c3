"""Runs of depthwise 3x3 -> 1x1 pairs as one kernel (sep_chain.cu), against the oracle and against the same network launched layer by
layer: ragged channels and planes, strides, one-sided pads, both orientations of the MMAs, with and without the classifier head,
one and several images per thread block."""
import pytest
import torch

from oracle import nets
from synth import configs
from synth.configs import P0, _conv, _fc, _gap
from paper_2303_04769_b200 import binding as B
from paper_2303_04769_b200.net import Net
from gpu_util import TOL, ctx, from_blk, pad_lanes_are_zero, rel_err, to_blk

pytestmark = pytest.mark.gpu


def run_of(C, H, W, pairs, head=None):
    """pairs: (filters, stride, pads, ReLU behind the depthwise layer, ReLU behind the 1x1 layer)."""
    layers, src, c, h, w = [], "in", C, H, W
    for i, (K, S, pad, mid, relu) in enumerate(pairs):
        dst = "out" if head is None and i == len(pairs) - 1 else f"p{i}"
        layers.append(dict(op="dwconv", name=f"d{i}", src=src, dst=f"m{i}", C=c, K=c, FH=3, FW=3, stride=S, pad=pad, relu=mid, accumulate=False))
        layers.append(_conv(f"c{i}", f"m{i}", dst, c, K, 1, 1, P0, relu))
        h, w = (h + pad[0] + pad[1] - 3) // S + 1, (w + pad[2] + pad[3] - 3) // S + 1
        src, c = dst, K
    if head is not None:
        layers += [_gap("gap", src, "g", c), _fc("fc", "g", "out", c, head)]
    return dict(name="run", batch=1, input=(C, H, W), input_dist=("uniform", -1.0, 1.0), weight_dist="he_normal", layers=layers)


SAME, HALF, NONE = (1, 1, 1, 1), (1, 0, 0, 1), (0, 0, 0, 0)
RUNS = {
    "one_pixel": run_of(8, 1, 1, [(9, 1, SAME, True, True)] * 1 + [(9, 1, SAME, True, True)] * 2, 3),
    "columns_5": run_of(64, 25, 5, [(64, 1, SAME, True, True)] * 4, 12),                            # pixels on M, all the way
    "columns_5_wide": run_of(100, 23, 5, [(70, 1, SAME, False, True), (128, 1, SAME, True, False), (128, 1, SAME, True, True)]),
    "ragged": run_of(33, 9, 7, [(65, 1, HALF, True, True), (31, 2, (2, 1, 1, 2), True, True), (40, 1, SAME, False, False)], 37),
    "px_16_edge": run_of(40, 16, 16, [(40, 2, SAME, True, True), (24, 2, SAME, True, True), (24, 1, SAME, True, True)]),
    "two_filter_tiles": run_of(128, 6, 6, [(256, 2, SAME, True, True), (200, 1, SAME, True, True), (129, 1, SAME, True, True)], 2),
    "plane_144": run_of(32, 24, 24, [(64, 2, SAME, True, True), (64, 1, SAME, True, True), (128, 2, SAME, True, True)]),
    "no_pads": run_of(48, 12, 12, [(48, 1, NONE, True, True), (48, 1, NONE, True, True), (48, 1, NONE, True, True)], 1),
    "growing_ring": run_of(64, 12, 12, [(64, 1, SAME, True, True), (128, 2, SAME, True, True), (128, 1, SAME, True, True), (128, 1, SAME, True, True), (256, 2, SAME, True, True)], 9),
}


@pytest.mark.parametrize("batch", [1, 5])
@pytest.mark.parametrize("math", ["tf32", "3xtf32"])
@pytest.mark.parametrize("name", RUNS)
def test_run_matches_the_oracle(name, math, batch):
    net = RUNS[name]
    params, x = configs.make_params(net), configs.make_input(net, batch)
    ref = nets.run_net(net, params, x)["out"]
    gnet = Net(ctx(), net, params, batch=batch, math=math)
    assert gnet.forms() == (["pair_run"] * len(net["layers"]), 1)
    got = gnet.run(to_blk(x))
    assert rel_err(from_blk(got, batch, *ref.shape[1:]), ref) <= TOL[math]
    assert pad_lanes_are_zero(got, batch, *ref.shape[1:])
    assert B.small_device_status(ctx()) == 0


@pytest.mark.parametrize("name,batch", [("columns_5", 149), ("columns_5", 700), ("ragged", 297), ("plane_144", 300), ("two_filter_tiles", 148), ("two_filter_tiles", 200), ("px_16_edge", 1100)])
@pytest.mark.parametrize("math", ["tf32", "3xtf32"])
def test_many_images_match_the_layers_one_by_one(name, math, batch):
    """Several images per thread block, two blocks per SM: the stream of filters crosses the images' ends.  Both forms round alike but
    for the order of sums, so they agree far inside the tolerance: FP32 sums of at most 256 products, 1e-5.  In TF32 such a difference
    can take an operand of the next layer across a rounding boundary: one product is then off by 2^-10 of its size, which is at most
    the MAX_ELEMENT_FACTOR = 8 rms that rel_err divides by."""
    net = RUNS[name]
    params, x = configs.make_params(net), configs.make_input(net, batch)
    blk = to_blk(x)
    gnet, apart = (Net(ctx(), net, params, batch=batch, math=math, **kw) for kw in ({}, dict(fuse_dwpw=False)))
    # (many filters on few pixels: layer by layer where images come in several rounds)
    assert (gnet.forms()[1] == 1) == ((name, batch, math) != ("two_filter_tiles", 200, "3xtf32")) and apart.forms()[1] >= len(net["layers"]) - 1
    shape = (batch,) + tuple(gnet.out_shape)
    want = from_blk(apart.run(blk), *shape)
    got = gnet.run(blk)
    assert rel_err(from_blk(got, *shape), want) <= (1e-5 if math == "3xtf32" else 2.0 ** -10)
    first = got.clone()
    for _ in range(3):
        assert torch.equal(gnet.run(blk), first)
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        out = gnet.run(blk)
    out.fill_(float("nan"))
    g.replay()
    assert torch.equal(out, first)
    assert B.small_device_status(ctx()) == 0


def test_a_result_that_is_read_again_stays():
    """A pair whose result another layer reads as well ends the run: the tensor has to be written."""
    net = RUNS["columns_5"]
    layers = [dict(L) for L in net["layers"][:8]]
    layers[-1]["dst"] = "p3"
    layers += [_conv("j", "p1", "out", 64, 64, 1, 1, P0, False), _conv("k", "p3", "out", 64, 64, 1, 1, P0, False, accumulate=True)]
    net = dict(net, layers=layers)
    params, x = configs.make_params(net), configs.make_input(net, 3)
    ref = nets.run_net(net, params, x)["out"]
    got = from_blk(Net(ctx(), net, params, batch=3, math="3xtf32").run(to_blk(x)), 3, *ref.shape[1:])
    assert rel_err(got, ref) <= TOL["3xtf32"]


@pytest.mark.parametrize("head", [False, True])
@pytest.mark.parametrize("math", ["tf32", "3xtf32"])
@pytest.mark.parametrize("C,H,W,K", [(64, 25, 5, 64), (64, 25, 5, 40), (40, 6, 7, 70)])      # pixels on M, with pad filters; filters on M
def test_values_without_a_number_pass_as_in_the_layers_one_by_one(C, H, W, K, math, head):
    """Layers without ReLU hand a NaN and an infinity on, and pad filters stay zero beside them."""
    net = run_of(C, H, W, [(K, 1, SAME, False, False)] * 3, 12 if head else None)
    params, x = configs.make_params(net), configs.make_input(net, 4)
    x[0, 3, 2, 1], x[2, C - 1, H - 1, 0] = float("nan"), float("inf")
    shape, got = None, []
    for kw in ({}, dict(fuse_dwpw=False)):
        gnet = Net(ctx(), net, params, batch=4, math=math, **kw)
        assert ("pair_run" in gnet.forms()[0]) == (not kw)
        shape = (4,) + tuple(gnet.out_shape)
        out = gnet.run(to_blk(x))
        assert pad_lanes_are_zero(out, *shape)
        got.append(torch.from_numpy(from_blk(out, *shape)))
    run, layers = got
    assert torch.equal(run.isnan(), layers.isnan()) and torch.equal(run.isinf(), layers.isinf())
    assert not run[1].isnan().any() and run[0].isnan().any() and not run[2].isfinite().all()


@pytest.mark.parametrize("math", ["tf32", "3xtf32"])
@pytest.mark.parametrize("C,K", [(64, 8), (40, 12), (100, 5)])
def test_layers_computed_in_fp32_are_no_part_of_a_run(C, K, math):
    """A 1x1 layer of so few products per pixel that it computes in FP32 whatever the mode keeps its bits: it ends a run."""
    batch = 600
    net = run_of(C, 8, 8, [(C, 1, SAME, True, True), (K, 1, SAME, True, True), (C, 1, SAME, True, True)])
    assert B.small_conv2d_path(ctx(), batch, C, K, 8, 8, 1, 1, 1, NONE, B.MATH[math]) in (1, 2)
    params, blk = configs.make_params(net), to_blk(configs.make_input(net, batch))
    run, apart = (Net(ctx(), net, params, batch=batch, math=math, **kw) for kw in ({}, dict(fuse_dwpw=False)))
    assert "pair_run" not in run.forms()[0]
    assert torch.equal(run.run(blk).clone(), apart.run(blk))
