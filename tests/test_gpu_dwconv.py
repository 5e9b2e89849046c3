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


@pytest.mark.parametrize("case", [(128, 64, 56, 56, 1), (96, 64, 25, 5, 1), (64, 128, 56, 56, 2), (200, 96, 7, 7, 1)])
def test_depthwise_3x3_repeats_its_bits(case):
    """A slot of the ring that were refilled while a lane still reads it would change bits now and then: the same layer some
    hundred times, back to back on a full chip, against its own first result (which the oracle checks on one image)."""
    N, C, H, W, S = case
    x, w, b = synth.uniform((N, C, H, W), -1, 1, 4, seed=77), synth.uniform((C, 3, 3), -1, 1, 5, seed=77), synth.uniform((C,), -1, 1, 6, seed=77)
    OH, OW = B.small_out_size(H, 3, S, 1, 1), B.small_out_size(W, 3, S, 1, 1)
    wb, bias = torch.empty(B.small_dw_weight_elems(C, 3, 3), device="cuda"), dev(b)
    B.small_pack_dw_weights(ctx(), dev(w), wb, C, 3, 3)
    xb = to_blk(x)
    out, first, wrong = new_blk(N, C, OH, OW), None, torch.zeros((), dtype=torch.int64, device="cuda")
    for i in range(400):
        out.fill_(float("nan"))
        B.small_dwconv2d(ctx(), xb, wb, bias, out, N, C, H, W, 3, 3, S, (1, 1, 1, 1), B.RELU)
        if first is None:
            first = out.clone()
        wrong += (out.view(torch.int32) != first.view(torch.int32)).sum()
    assert int(wrong) == 0
    n = N // 2
    assert rel_err(from_blk(first, N, C, OH, OW)[n:n + 1], oracle.dwconv2d(x[n:n + 1], w, b, S, (1, 1, 1, 1), True)) <= 1e-5
    assert B.small_device_status(ctx()) == 0
