"""Layers of few output pixels in the tensor-core modes: the reduction of a tile split over warps, at the edges of tiles, filter
blocks and splits, against the oracle; with the pad lanes, the join and an output that is only 16-byte aligned."""
import pytest
import torch

import oracle
import synth
from paper_2303_04769_b200 import binding as B
from gpu_util import ctx, dev, to_blk, from_blk, rel_err, pad_lanes_are_zero, conv_path

pytestmark = pytest.mark.gpu
TOL = {"tf32": 2e-3, "3xtf32": 1e-5}

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


@pytest.mark.parametrize("math", ["tf32", "3xtf32"])
@pytest.mark.parametrize("case", CASES)
def test_few_pixels(case, math):
    N, C, K, H, W, FH, FW, S, pad = case
    m = B.MATH[math]
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


def test_split_sums_are_closer_than_one_chain():
    N, C, K, H = 1, 256, 64, 7
    x, w = synth.uniform((N, C, H, H), -1, 1, 1, seed=3), synth.uniform((K, C, 3, 3), -1, 1, 2, seed=3)
    ref = oracle.conv2d(x, w, None, 1, (1, 1, 1, 1))
    wb = torch.empty(B.small_conv_weight_elems(C, K, 3, 3, B.MATH_3XTF32), device="cuda")
    B.small_pack_conv_weights(ctx(), dev(w), wb, C, K, 3, 3, B.MATH_3XTF32)

    def err():
        out = torch.empty(B.small_packed_elems(N, K, H, H), device="cuda")
        B.small_conv2d(ctx(), to_blk(x), wb, None, out, N, C, K, H, H, 3, 3, 1, (1, 1, 1, 1), B.MATH_3XTF32)
        return rel_err(from_blk(out, N, K, H, H), ref)

    split = err()
    with conv_path("tensor"):
        assert split < err()        # 144 steps of one accumulator against 9 of 16
