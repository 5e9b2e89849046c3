"""Which tensor-core kernel a 3x3 layer of 17 to 32 channels and filters and a 1x1 layer of up to 64 filters goes to, at the
edges of the rules, and its result."""
import pytest
import torch

import oracle
import synth
from paper_2303_04769_b200 import binding as B
from gpu_util import ctx, dev, to_blk, from_blk, new_blk, rel_err, pad_lanes_are_zero

pytestmark = pytest.mark.gpu
BLOCK, WARP = 3, 4
TOL = {"tf32": 2e-3, "3xtf32": 1e-5}

CASES = [  # math, window, N, C, K, H, W, kernel
    ("3xtf32", 3, 1, 17, 17, 5, 5, BLOCK),
    ("3xtf32", 3, 1, 16, 32, 5, 5, WARP),
    ("3xtf32", 3, 1, 32, 16, 16, 16, WARP),
    ("3xtf32", 3, 2, 32, 32, 3, 72, BLOCK),
    ("3xtf32", 3, 2, 32, 32, 3, 73, WARP),
    ("tf32", 3, 111, 24, 32, 30, 30, WARP),
    ("tf32", 3, 112, 24, 32, 30, 30, BLOCK),
    ("tf32", 3, 1, 32, 32, 16, 16, WARP),     # one image: cut into as many tiles as its warps can be dealt
    ("3xtf32", 3, 1, 16, 16, 13, 31, WARP),
    ("tf32", 1, 32, 20, 40, 32, 32, BLOCK),
    ("3xtf32", 1, 32, 32, 64, 32, 32, BLOCK),
    ("3xtf32", 1, 31, 32, 64, 32, 32, WARP),
    ("tf32", 1, 32, 16, 64, 32, 32, WARP),
    ("tf32", 1, 32, 32, 32, 32, 32, WARP),
]


@pytest.mark.parametrize("case", CASES)
def test_layers_of_one_channel_block(case):
    math, F, N, C, K, H, W, kernel = case
    m, pad = B.MATH[math], (F // 2,) * 4
    x, w, b = synth.uniform((N, C, H, W), -1, 1, 1, seed=5), synth.uniform((K, C, F, F), -1, 1, 2, seed=5), synth.uniform((K,), -1, 1, 3, seed=5)
    assert B.small_conv2d_path(ctx(), N, C, K, H, W, F, F, 1, pad, m) == kernel
    wb = torch.empty(B.small_conv_weight_elems(C, K, F, F, m), device="cuda")
    B.small_pack_conv_weights(ctx(), dev(w), wb, C, K, F, F, m)
    out = new_blk(N, K, H, W)
    B.small_conv2d(ctx(), to_blk(x), wb, dev(b), out, N, C, K, H, W, F, F, 1, pad, B.RELU | m)
    assert rel_err(from_blk(out, N, K, H, W), oracle.conv2d(x, w, b, 1, pad, relu=True)) <= TOL[math]
    assert pad_lanes_are_zero(out, N, K, H, W)
