"""The fused chain of full reductions where its stages and operand slots end unevenly: odd numbers of channel blocks in the first, a
middle and the last layer, a first layer that goes through the slots several times, and several tiles per thread block."""
import pytest
import torch

import oracle
import synth
from paper_2303_04769_b200 import binding as B
from gpu_util import TOL, ctx, dev, from_blk, new_blk, pad_lanes_are_zero, rel_err, to_blk

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("widths,N,tile", [
    ([288, 96, 65, 8, 160], 100, 0), ([545, 128, 40], 70, 0), ([1000, 7, 90, 128, 513], 33, 0), ([8, 8, 8], 1, 0),
    ([640, 128, 96, 128, 300], 5000, 32), ([95, 128, 70, 128], 9600, 32), ([320, 64, 32], 9500, 64), ([160, 128, 129], 19100, 128)])
@pytest.mark.parametrize("math", ["tf32", "3xtf32"])
def test_uneven_stages(widths, N, tile, math):
    L = len(widths) - 1
    ws = [synth.he_normal((widths[i + 1], widths[i]), widths[i], 500 + 2 * i, 3) for i in range(L)]
    bs = [synth.uniform((widths[i + 1],), -0.1, 0.1, 501 + 2 * i, 3) for i in range(L)]
    x = synth.normal((N, widths[0], 1, 1), 0.0, 1.0, 499, 3)
    wbs = []
    for i, w in enumerate(ws):
        wb = torch.empty(B.small_fc_weight_elems(widths[i], widths[i + 1], B.MATH[math]), device="cuda")
        B.small_pack_fc_weights(ctx(), dev(w), wb, widths[i], widths[i + 1], B.MATH[math])
        wbs.append(wb)
    dbs, relu, bx, out = [dev(b) for b in bs], [i != L - 1 for i in range(L)], to_blk(x), new_blk(N, widths[-1], 1, 1)
    try:
        B.small_set_fc_chain_tile(ctx(), tile)
        B.small_fc_chain(ctx(), bx, wbs, dbs, widths, relu, out, None, N, B.MATH[math])
        got = from_blk(out, N, widths[-1], 1, 1).reshape(N, widths[-1])
    finally:
        B.small_set_fc_chain_tile(ctx(), 0)
    assert B.small_device_status(ctx()) == 0
    pick = list(range(min(N, 40))) + list(range(max(0, N - 40), N))      # both ends: the oracle takes an image at a time
    ref = x.reshape(N, widths[0])[pick]
    for w, b, r in zip(ws, bs, relu):
        ref = oracle.fc(ref, w, b, relu=r)
    assert rel_err(got[pick], ref) <= 2.5 * TOL[math]                    # a chain compounds each layer's rounding
    assert pad_lanes_are_zero(out, N, widths[-1], 1, 1)
