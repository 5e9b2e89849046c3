"""The few-input-channel kernel at the edges of its tiles: every number of lanes per filter group, rows cut into bands, several images
per tile, planes too wide for one TMA box, and the network's NCHW edge."""
import numpy as np
import pytest
import torch

import oracle
import synth
from synth import configs
from paper_2303_04769_b200 import binding as B
from paper_2303_04769_b200.net import Net
from gpu_util import ctx, dev, from_blk, new_blk, pad_lanes_are_zero, rel_err, to_blk

pytestmark = pytest.mark.gpu

P1 = (1, 1, 1, 1)
CASES = [  # N, C, K, H, W, FH, FW, stride, pad
    (2, 2, 1, 6, 17, 3, 3, 1, P1), (3, 3, 9, 8, 8, 3, 3, 2, P1), (2, 1, 17, 20, 31, 3, 3, 1, P1), (2, 4, 64, 15, 16, 3, 3, 1, P1),
    (1, 3, 96, 33, 33, 3, 3, 2, P1), (2, 1, 65, 49, 10, 10, 4, 2, (4, 5, 1, 1)), (90, 2, 24, 7, 5, 3, 3, 1, P1), (400, 1, 48, 14, 10, 10, 4, 2, (4, 5, 1, 1)),
    (2, 1, 8, 5, 300, 3, 3, 1, P1), (1, 4, 33, 9, 511, 3, 3, 2, P1), (1, 1, 40, 30, 260, 10, 4, 2, (0, 0, 0, 0)), (1, 1, 16, 700, 9, 3, 3, 1, P1),
    (150, 3, 16, 4, 4, 3, 3, 2, (0, 1, 0, 1)),
]


@pytest.mark.parametrize("case", CASES)
def test_tiles_match_the_oracle(case):
    N, C, K, H, W, FH, FW, S, pad = case
    x, w, b = (synth.uniform(s, -1.0, 1.0, t) for s, t in (((N, C, H, W), 81), ((K, C, FH, FW), 82), ((K,), 83)))
    wb = torch.empty(B.small_conv_weight_elems(C, K, FH, FW, B.MATH_FP32), device="cuda")
    B.small_pack_conv_weights(ctx(), dev(w), wb, C, K, FH, FW, B.MATH_FP32)
    ref = oracle.conv2d(x, w, b, S, pad, relu=True)
    out = new_blk(N, K, *ref.shape[2:])
    for _ in range(2):                       # the second call takes the finished launch
        out.fill_(float("nan"))
        B.small_conv2d(ctx(), to_blk(x), wb, dev(b), out, N, C, K, H, W, FH, FW, S, pad, B.RELU)
        assert rel_err(from_blk(out, N, K, *ref.shape[2:]), ref) <= 1e-5      # FP32 sums of at most 40 products
        assert pad_lanes_are_zero(out, N, K, *ref.shape[2:])
    assert B.small_device_status(ctx()) == 0


@pytest.mark.parametrize("name,batch", [("kws_cnn", 1), ("kws_cnn", 333), ("dwsep_cnn", 3), ("residual_cnn", 70)])
def test_nchw_and_blocked_inputs_give_the_same_bits(name, batch):
    net = configs.NETWORKS[name](batch=batch)
    x = configs.make_input(net, batch)
    gnet = Net(ctx(), net, configs.make_params(net), batch=batch, math="tf32")
    host = torch.full((batch,) + tuple(gnet.out_shape), float("nan")).pin_memory()
    gnet.run_host(torch.from_numpy(x).pin_memory(), host)
    torch.cuda.synchronize()
    np.testing.assert_array_equal(host.numpy(), from_blk(gnet.run(to_blk(x)), batch, *gnet.out_shape))


WIDE = [  # planes whose rows are cut into column bands: one channel to four, every window; last bands of one column group and of a few columns
    (1, 1, 16, 8, 3300, 3, 3, 1, P1), (1, 1, 16, 8, 1680, 3, 3, 1, P1), (1, 3, 16, 1000, 1000, 3, 3, 1, P1), (1, 3, 9, 672, 672, 3, 3, 2, P1),
    (2, 4, 70, 19, 720, 3, 3, 2, (0, 1, 0, 1)), (1, 2, 24, 840, 840, 3, 3, 2, P1), (1, 1, 40, 600, 1000, 10, 4, 2, (4, 5, 1, 1)), (1, 4, 5, 448, 448, 3, 3, 2, P1),
    (3, 3, 33, 5, 225, 3, 3, 1, (2, 0, 2, 0)), (1, 3, 64, 7, 265, 3, 3, 1, (0, 0, 0, 0)), (1, 4, 8, 3, 851, 3, 3, 1, (0, 0, 0, 0)),
]


@pytest.mark.parametrize("case", WIDE)
def test_wide_planes_match_the_oracle(case):
    """Rows too long for a tile of whole ones (a tile of one row was more than a block's shared memory for some of these widths)."""
    test_tiles_match_the_oracle(case)


@pytest.mark.parametrize("C,H,W,S", [(3, 30, 672, 2), (1, 9, 1680, 1), (4, 40, 300, 1)])
def test_wide_planes_from_nchw_give_the_same_bits(C, H, W, S):
    layers = [configs._conv("stem", "in", "a", C, 20, 3, S, P1, True), configs._conv("p", "a", "out", 20, 8, 1, 1, configs.P0, False)]
    net = dict(name="wide", batch=2, input=(C, H, W), input_dist=("uniform", -1.0, 1.0), weight_dist="he_normal", layers=layers)
    x = configs.make_input(net, 2)
    gnet = Net(ctx(), net, configs.make_params(net), batch=2)
    host = torch.full((2,) + tuple(gnet.out_shape), float("nan")).pin_memory()
    gnet.run_host(torch.from_numpy(x).pin_memory(), host)
    torch.cuda.synchronize()
    np.testing.assert_array_equal(host.numpy(), from_blk(gnet.run(to_blk(x)), 2, *gnet.out_shape))
