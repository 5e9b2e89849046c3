"""Layers of few output pixels: the reduction of a tile split over warps, on the tensor cores and in FP32, at the edges of tiles, filter
blocks and splits, against the oracle; with the pad lanes, the join and an output that is only 16-byte aligned."""
import pytest
import torch

import oracle
import synth
from oracle import nets
from paper_2303_04769_b200 import binding as B
from paper_2303_04769_b200.net import Net
from synth import configs
from gpu_util import ctx, dev, to_blk, from_blk, rel_err, pad_lanes_are_zero, conv_path

pytestmark = pytest.mark.gpu
TOL = {"fp32": 1e-5, "tf32": 2e-3, "3xtf32": 1e-5}

CASES = [  # N, C, K, H, W, FH, FW, stride, pad (t, b, l, r)
    (1, 16, 16, 32, 32, 3, 3, 1, (1, 1, 1, 1)),
    (1, 17, 17, 5, 5, 3, 3, 1, (1, 1, 1, 1)),
    (3, 16, 41, 5, 7, 3, 3, 2, (0, 1, 1, 0)),       # pixels of three images in one tile, filters behind the last tile
    (1, 8, 64, 1, 1, 1, 1, 1, (0, 0, 0, 0)),        # one pixel, one step
    (2, 300, 9, 4, 4, 1, 1, 1, (0, 0, 0, 0)),
    (1, 70, 33, 9, 8, 3, 3, 1, (2, 0, 0, 2)),
    (5, 33, 130, 6, 5, 3, 3, 2, (1, 1, 1, 1)),
    (1, 512, 96, 5, 5, 3, 3, 1, (1, 1, 1, 1)),
    (7, 64, 64, 8, 8, 3, 3, 1, (1, 1, 1, 1)),
]


@pytest.mark.parametrize("math", ["fp32", "tf32", "3xtf32"])
@pytest.mark.parametrize("case", CASES)
def test_few_pixels(case, math):
    N, C, K, H, W, FH, FW, S, pad = case
    m = B.MATH[math]
    # (one step on one pixel in TF32 is as fast as a whole tile)
    assert B.small_conv2d_split(ctx(), N, C, K, H, W, FH, FW, S, pad, m) == (not (math == "tf32" and (C, H) == (8, 1)))
    x, w, b = synth.uniform((N, C, H, W), -1, 1, 1, seed=9), synth.uniform((K, C, FH, FW), -1, 1, 2, seed=9), synth.uniform((K,), -1, 1, 3, seed=9)
    ref = oracle.conv2d(x, w, b, S, pad, relu=True)
    OH, OW = ref.shape[2:]
    wb = torch.empty(B.small_conv_weight_elems(C, K, FH, FW, m), device="cuda")
    B.small_pack_conv_weights(ctx(), dev(w), wb, C, K, FH, FW, m)
    n = B.small_packed_elems(N, K, OH, OW)
    room = torch.full((n + 72,), float("nan"), device="cuda")
    for start in (32, 36):                          # 36: not a multiple of 32 bytes
        room.fill_(float("nan"))
        out = room[start:start + n]
        B.small_conv2d(ctx(), to_blk(x), wb, dev(b), out, N, C, K, H, W, FH, FW, S, pad, B.RELU | m)
        assert rel_err(from_blk(out, N, K, OH, OW), ref) <= TOL[math]
        assert pad_lanes_are_zero(out, N, K, OH, OW)
        assert room[:start].isnan().all() and room[start + n:].isnan().all()
    prev = synth.uniform((N, K, OH, OW), -1, 1, 4, seed=9)
    acc = to_blk(prev)
    B.small_conv2d(ctx(), to_blk(x), wb, None, acc, N, C, K, H, W, FH, FW, S, pad, B.ACCUMULATE | m)
    assert rel_err(from_blk(acc, N, K, OH, OW), oracle.conv2d(x, w, None, S, pad, accumulate_into=prev)) <= TOL[math]
    assert pad_lanes_are_zero(acc, N, K, OH, OW)


@pytest.mark.parametrize("math", ["fp32", "tf32", "3xtf32"])
def test_values_without_a_number_stay_where_they_are(math):
    """An infinite or missing input reaches the pixels whose window holds it and no other, and no pad filter.  (3xTF32: the residual of an
    infinity is no number.)"""
    m = B.MATH[math]
    assert B.small_conv2d_split(ctx(), 1, 40, 33, 9, 9, 3, 3, 1, (1, 1, 1, 1), m) == 1
    x, w = synth.uniform((1, 40, 9, 9), -1, 1, 1, seed=4), abs(synth.uniform((33, 40, 3, 3), -1, 1, 2, seed=4)) + 0.1
    x[0, 3, 0, 0], x[0, 39, 8, 4] = float("inf"), float("nan")
    wb = torch.empty(B.small_conv_weight_elems(40, 33, 3, 3, m), device="cuda")
    B.small_pack_conv_weights(ctx(), dev(w), wb, 40, 33, 3, 3, m)
    out = torch.empty(B.small_packed_elems(1, 33, 9, 9), device="cuda")
    B.small_conv2d(ctx(), to_blk(x), wb, None, out, 1, 40, 33, 9, 9, 3, 3, 1, (1, 1, 1, 1), m)
    assert pad_lanes_are_zero(out, 1, 33, 9, 9)
    got = torch.from_numpy(from_blk(out, 1, 33, 9, 9))
    want = torch.nn.functional.conv2d(torch.from_numpy(x).double(), torch.from_numpy(w).double(), padding=1)
    assert torch.equal(got.isfinite(), want.isfinite()) and (~want.isfinite()).sum() == 33 * 10
    if math != "3xtf32":
        assert torch.equal(got.isinf(), want.isinf()) and torch.equal(got.isnan(), want.isnan())
        assert got.isinf().sum() == 33 * 4 and got.isnan().sum() == 33 * 6


@pytest.mark.parametrize("math,path", [("3xtf32", "tensor"), ("fp32", "cuda_cores")])
def test_split_sums_are_closer_than_one_chain(math, path):
    N, C, K, H, m = 1, 256, 64, 7, B.MATH[math]
    x, w = synth.uniform((N, C, H, H), -1, 1, 1, seed=3), synth.uniform((K, C, 3, 3), -1, 1, 2, seed=3)
    ref = oracle.conv2d(x, w, None, 1, (1, 1, 1, 1))
    wb = torch.empty(B.small_conv_weight_elems(C, K, 3, 3, m), device="cuda")
    B.small_pack_conv_weights(ctx(), dev(w), wb, C, K, 3, 3, m)

    def err():
        out = torch.empty(B.small_packed_elems(N, K, H, H), device="cuda")
        B.small_conv2d(ctx(), to_blk(x), wb, None, out, N, C, K, H, H, 3, 3, 1, (1, 1, 1, 1), m)
        return rel_err(from_blk(out, N, K, H, H), ref)

    split = err()
    with conv_path(path):
        assert split < err()        # a chain of 2304 products (288 steps of 8) against 16 of a sixteenth


@pytest.mark.parametrize("C,K,H,W,S,relu,batch", [(64, 64, 25, 5, 1, True, 2), (33, 70, 9, 7, 2, False, 3), (8, 24, 1, 1, 1, True, 1), (100, 9, 6, 5, 2, True, 4)])
def test_fp32_pairs_as_one_launch(C, K, H, W, S, relu, batch):
    """A depthwise 3x3 and a 1x1 layer of a small batch in FP32: ragged channels and planes, strides, one pixel."""
    layers = [dict(op="dwconv", name="d", src="in", dst="m", C=C, K=C, FH=3, FW=3, stride=S, pad=(1, 1, 1, 1), relu=relu, accumulate=False),
              configs._conv("c", "m", "out", C, K, 1, 1, configs.P0, True)]
    net = dict(name="pair", batch=batch, input=(C, H, W), input_dist=("uniform", -1.0, 1.0), weight_dist="he_normal", layers=layers)
    params, x = configs.make_params(net), configs.make_input(net, batch)
    ref = nets.run_net(net, params, x)["out"]
    gnet = Net(ctx(), net, params, batch=batch)
    assert gnet.forms() == (["pair_fp32"] * 2, 1)
    got = gnet.run(to_blk(x))
    assert rel_err(from_blk(got, *ref.shape), ref) <= TOL["fp32"]
    assert pad_lanes_are_zero(got, *ref.shape)
    apart = Net(ctx(), net, params, batch=batch, fuse_dwpw=False).run(to_blk(x))
    assert rel_err(from_blk(apart, *ref.shape), ref) <= TOL["fp32"]


@pytest.mark.parametrize("math", ["fp32", "tf32", "3xtf32"])
@pytest.mark.parametrize("C,K,H,W,C2,S,relu,batch", [(32, 32, 16, 16, 16, 2, True, 1), (12, 40, 7, 5, 70, 1, False, 3), (16, 9, 1, 1, 33, 3, True, 1), (64, 64, 8, 8, 32, 2, True, 2)])
def test_shortcut_as_part_of_the_layer_it_joins(math, C, K, H, W, C2, S, relu, batch):
    """x -> 1x1 shortcut (stride S) and 3x3 convolution, then a 3x3 convolution added to the shortcut: one launch for the last two."""
    H2, W2 = (H - 1) * S + 1 + (S > 2), (W - 1) * S + 1
    layers = [configs._conv("a", "in", "m", C2, C, 1, S, configs.P0, True),
              configs._conv("s", "in", "out", C2, K, 1, S, configs.P0, False),
              configs._conv("b", "m", "out", C, K, 3, 1, configs.P1, relu, accumulate=True)]
    net = dict(name="joined", batch=batch, input=(C2, H2, W2), input_dist=("uniform", -1.0, 1.0), weight_dist="he_normal", layers=layers)
    params, x = configs.make_params(net), configs.make_input(net, batch)
    ref = nets.run_net(net, params, x)["out"]
    # (33 -> 9: a 1x1 layer of few products computes in FP32 in every mode, its 3x3 does not)
    forms, launches = Net(ctx(), net, params, batch=batch, math=math).forms()
    assert (forms, launches) == ((["layer", "joined", "joined"], 2) if math == "fp32" or C2 != 33 else (["side_by_side"] * 2 + ["layer"], 3))
    for overlap in (1, 0):
        B.small_set_layer_overlap(ctx(), overlap)
        try:
            got = Net(ctx(), net, params, batch=batch, math=math).run(to_blk(x))
            apart = Net(ctx(), net, params, batch=batch, math=math, fuse_poolfc=False).run(to_blk(x))
        finally:
            B.small_set_layer_overlap(ctx(), 1)
        for y in (got, apart):
            assert rel_err(from_blk(y, *ref.shape), ref) <= TOL[math]
            assert pad_lanes_are_zero(y, *ref.shape)
