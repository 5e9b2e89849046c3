"""Runs of layers kept on chip as one kernel, against the oracle and against the same network launched layer by layer: ragged
channel counts and planes, strides, residual joins, one to eight thread blocks per image."""
import numpy as np
import pytest
import torch

from oracle import nets
from synth import configs
from synth.configs import P0, P1, _conv, _dw, _fc, _gap
from paper_2303_04769_b200 import binding as B
from paper_2303_04769_b200.net import Net
from gpu_util import TOL, ctx, from_blk, rel_err, to_blk

pytestmark = pytest.mark.gpu


def separable(H, W, C, K):
    """Depthwise and 1x1 layers whose channels are no multiples of anything, a 3x3 behind them, a strided pair."""
    L = [_conv("c0", "in", "a", C, K, 1, 1, P0, True), _dw("d1", "a", "b", K, 1), _conv("p1", "b", "c", K, C, 1, 1, P0, True),
         _dw("d2", "c", "d", C, 2), _conv("p2", "d", "e", C, K + 9, 1, 1, P0, True), _conv("c3", "e", "f", K + 9, 24, 3, 1, P1, True),
         _gap("gap", "f", "g", 24), _fc("fc", "g", "out", 24, 37)]
    return dict(name="separable", batch=1, input=(C, H, W), input_dist=("uniform", -1.0, 1.0), weight_dist="he_normal", layers=L)


def joined():
    """A residual join and a strided shortcut without depthwise layers."""
    L = [_conv("a", "in", "x", 20, 12, 3, 1, P1, True), _conv("b", "x", "y", 12, 40, 3, 2, P1, True), _conv("s", "x", "z", 12, 40, 1, 2, P0, False),
         _conv("c", "y", "z", 40, 40, 3, 1, P1, True, accumulate=True), _gap("gap", "z", "g", 40), _fc("fc", "g", "out", 40, 5)]
    return dict(name="joined", batch=1, input=(20, 13, 11), input_dist=("uniform", -1.0, 1.0), weight_dist="he_normal", layers=L)


@pytest.mark.parametrize("math", ["fp32", "tf32", "3xtf32"])
@pytest.mark.parametrize("net,batch", [(separable(9, 7, 20, 33), 1), (separable(6, 16, 40, 64), 30), (separable(5, 5, 8, 100), 70),
                                       (separable(11, 3, 33, 17), 148), (joined(), 3)])
def test_on_chip_runs_match(net, batch, math):
    params = configs.make_params(net)
    x = configs.make_input(net, batch)
    ref = nets.run_net(net, params, x)["out"]
    blk = to_blk(x)
    gnet = Net(ctx(), net, params, batch=batch, math=math)
    # (FP32 at small batches and networks without depthwise layers run launch by launch)
    assert (gnet.forms()[1] == 1) == (math != "fp32" and net["name"] == "separable")
    got = from_blk(gnet.run(blk), batch, *ref.shape[1:])
    apart = from_blk(Net(ctx(), net, params, batch=batch, math=math, fuse_poolfc=False).run(blk), batch, *ref.shape[1:])
    assert rel_err(got, ref) <= TOL[math] and rel_err(apart, ref) <= TOL[math]
    assert B.small_device_status(ctx()) == 0


@pytest.mark.parametrize("batch", [3, 100])
def test_result_in_the_slot_of_the_runs_input(batch):
    """A list may end in the slot that its last layers' input came from: images do not wait for one another on chip, so the run has
    to start at a later layer, which reads another slot."""
    net = configs.kws_cnn(batch=batch)
    params, blk = configs.make_params(net), to_blk(configs.make_input(net, batch))
    gnet = Net(ctx(), net, params, batch=batch)
    want = gnet.run(blk).clone()
    last = len(gnet.layers) - 1
    slot = 1 + max(L.dst for L in gnet.layers)
    gnet.layers[0].dst = gnet.layers[1].src = gnet.layers[last].dst = slot
    size = B.small_net_workspace_bytes(gnet.layers, batch)
    workspace = torch.empty(size + 256, dtype=torch.uint8, device="cuda")
    assert ("on_chip" in B.small_net_forms(ctx(), gnet.layers, batch)[0]) == (batch == 100)
    start = size - (B.small_packed_elems(batch, 64, 25, 5) * 4 + 255) // 256 * 256          # the last slot, as large as the input
    for _ in range(20):
        workspace[start:].fill_(255)
        B.small_run_net(ctx(), gnet.layers, batch, blk, gnet.out_blk, workspace, size)
        got = workspace[start:start + 4 * want.numel()].view(torch.float32)
        assert rel_err(from_blk(got, batch, *gnet.out_shape), from_blk(want, batch, *gnet.out_shape)) <= TOL["fp32"]


@pytest.mark.parametrize("batch,math,form", [(40, "3xtf32", "pair_run"), (100, "fp32", "on_chip"), (148, "fp32", "on_chip")])
def test_on_chip_run_repeats_its_bits_in_a_graph(batch, math, form):
    net = configs.kws_cnn(batch=batch)
    gnet = Net(ctx(), net, configs.make_params(net), math=math)
    assert form in gnet.forms()[0]
    blk = to_blk(configs.make_input(net))
    want = gnet.run(blk).clone()
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        out = gnet.run(blk)
    for _ in range(3):
        out.fill_(float("nan"))
        g.replay()
        assert torch.equal(out, want)


def stack(C, n):
    L = [_conv("stem", "in", "p0", 1, C, (10, 4), 2, (4, 5, 1, 1), True)]
    for i in range(n):
        L += [_dw(f"d{i}", f"p{i}", f"m{i}", C, 1), _conv(f"c{i}", f"m{i}", f"p{i + 1}", C, C, 1, 1, P0, True)]
    L += [_gap("gap", f"p{n}", "g", C), _fc("fc", "g", "out", C, 12)]
    return dict(name="stack", batch=1, input=(1, 49, 10), input_dist=("normal", 0.0, 1.0), weight_dist="he_normal", layers=L)


@pytest.mark.parametrize("net,batch,math", [
    (stack(64, 3), 148, "fp32"), (stack(48, 4), 100, "fp32"), (stack(128, 4), 30, "fp32"), (stack(128, 2), 74, "fp32"), (stack(64, 1), 18, "3xtf32"), (stack(64, 2), 30, "3xtf32"),
    (stack(24, 1), 1, "tf32"), (separable(11, 3, 33, 17), 2, "tf32"), (separable(11, 3, 33, 17), 2, "3xtf32"), (separable(9, 7, 20, 33), 19, "3xtf32")])
def test_blocks_per_image_in_every_mode(net, batch, math):
    """One, two, four and eight thread blocks to an image, as far as each mode comes to the on-chip kernel."""
    params, x = configs.make_params(net), configs.make_input(net, batch)
    gnet = Net(ctx(), net, params, batch=batch, math=math)
    assert gnet.forms()[0][-4:] == ["on_chip"] * 4
    ref = nets.run_net(net, params, x)["out"]
    assert rel_err(from_blk(gnet.run(to_blk(x)), batch, *ref.shape[1:]), ref) <= TOL[math]
    assert B.small_device_status(ctx()) == 0


@pytest.mark.parametrize("C,batch,math,form", [(64, 9, "fp32", "pair_fp32"), (64, 100, "fp32", "on_chip"), (64, 148, "3xtf32", "on_chip"), (64, 60, "tf32", "on_chip"), (48, 9, "tf32", "on_chip"),
                                                  (64, 9, "3xtf32", "layer"), (96, 148, "tf32", "layer"), (128, 9, "3xtf32", "layer"),
                                                  (96, 9, "fp32", "pair_fp32"), (96, 60, "fp32", "layer"), (128, 148, "fp32", "layer"), (160, 9, "fp32", "layer")])
def test_which_runs_stay_on_chip(C, batch, math, form):
    """Either side of the lines between the forms.  The on-chip kernel and the pairs of few pixels add up in another order, so a result has
    the bits of the layers launched one by one exactly where those run."""
    net = stack(C, 2)
    params, x = configs.make_params(net), configs.make_input(net, batch)
    blk = to_blk(x)
    gnet = Net(ctx(), net, params, batch=batch, math=math)
    assert set(gnet.forms()[0][1:5]) == {form}
    got = gnet.run(blk)
    apart = Net(ctx(), net, params, batch=batch, math=math, fuse_dwpw=False).run(blk)
    assert torch.equal(got, apart) == (form == "layer")
    ref = nets.run_net(net, params, x)["out"]
    assert rel_err(from_blk(got, batch, *ref.shape[1:]), ref) <= TOL[math]
