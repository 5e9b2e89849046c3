"""GPU parity of the streamed depthwise 3x3 kernel where it changes shape: one to several bands of columns, odd last pairs,
sets of images that do not divide the batch, blocks that begin inside a plane, rings that wrap, changing filters."""
import pytest
import torch

import oracle
import synth
from paper_2303_04769_b200 import binding as B
from gpu_util import ctx, dev, to_blk, from_blk, new_blk, rel_err, pad_lanes_are_zero

pytestmark = pytest.mark.gpu

CASES = [  # N, C, H, W, S, pad
    (1, 32, 5, 2, 1, (1, 1, 1, 1)),        # one pair of columns
    (70, 5, 3, 1, 1, (1, 1, 1, 1)),        # half a pair; 32 images to a row, 70 of them
    (1, 3, 9, 64, 1, (1, 1, 1, 1)),        # one full band
    (1, 3, 9, 65, 1, (1, 1, 1, 1)),        # two bands, the last pair half empty
    (2, 33, 6, 131, 2, (0, 1, 1, 0)),      # two bands of stride 2, odd, padded on some sides
    (1, 8, 40, 224, 1, (1, 1, 1, 1)),      # four bands
    (9, 64, 7, 7, 1, (1, 1, 1, 1)),        # eight images to a row and one over
    (3, 40, 300, 9, 1, (2, 0, 0, 2)),      # long columns, blocks that begin inside a plane
    (48, 70, 31, 33, 2, (1, 1, 1, 1)),     # many rows to a block: the ring wraps, planes and filters change
    (33, 96, 28, 28, 1, (1, 1, 1, 1)),
]


@pytest.mark.parametrize("case", CASES)
def test_depthwise_3x3(case):
    N, C, H, W, S, pad = case
    x, w, b = synth.uniform((N, C, H, W), -1, 1, 1, seed=77), synth.uniform((C, 3, 3), -1, 1, 2, seed=77), synth.uniform((C,), -1, 1, 3, seed=77)
    ref = oracle.dwconv2d(x, w, b, S, pad, True)
    OH, OW = ref.shape[2:]
    wb = torch.empty(B.small_dw_weight_elems(C, 3, 3), device="cuda")
    B.small_pack_dw_weights(ctx(), dev(w), wb, C, 3, 3)
    xb = to_blk(x)
    for _ in range(2):                     # planned, and from the kept plan
        out = new_blk(N, C, OH, OW)
        out.fill_(float("nan"))
        B.small_dwconv2d(ctx(), xb, wb, dev(b), out, N, C, H, W, 3, 3, S, pad, B.RELU)
        assert rel_err(from_blk(out, N, C, OH, OW), ref) <= 1e-5
        assert pad_lanes_are_zero(out, N, C, OH, OW)
