"""The register-tiled FP32 convolution's tilings at their edges against the oracle: runs of 7 pixels (planes of 7, 14, 28 columns
and remainders), pointwise planes viewed with other row lengths, both filter tiles, several images per warp."""
import numpy as np
import pytest
import torch

import oracle
from paper_2303_04769_b200 import binding as B
from gpu_util import conv_path, ctx, dev, from_blk, new_blk, pad_lanes_are_zero, rel_err, to_blk

pytestmark = pytest.mark.gpu

CASES = [  # N, C, K, H, W, F, S, pad, accumulate
    (3, 40, 70, 14, 14, 3, 1, (1, 1, 1, 1), False),
    (9, 16, 64, 7, 7, 3, 1, (1, 1, 1, 1), True),
    (2, 33, 33, 28, 28, 3, 1, (1, 1, 1, 1), False),
    (2, 8, 96, 15, 29, 3, 1, (0, 1, 1, 0), False),      # a pixel more than whole runs
    (1, 20, 24, 5, 6, 3, 1, (1, 1, 1, 1), False),
    (11, 64, 64, 25, 5, 1, 1, (0, 0, 0, 0), True),      # rows of 125
    (1, 48, 40, 31, 29, 1, 1, (0, 0, 0, 0), False),
    (5, 128, 256, 3, 3, 1, 1, (0, 0, 0, 0), False),
    (2, 32, 48, 13, 11, 1, 2, (0, 0, 0, 0), False),
]


@pytest.mark.parametrize("case", CASES)
def test_conv_direct_tilings(case):
    N, C, K, H, W, F, S, pad, acc = case
    rng = np.random.RandomState(31)
    x, w = rng.uniform(-1, 1, (N, C, H, W)).astype(np.float32), rng.uniform(-1, 1, (K, C, F, F)).astype(np.float32)
    b = rng.uniform(-1, 1, K).astype(np.float32)
    ref = oracle.conv2d(x, w, b, S, pad, relu=False)
    prev = rng.uniform(-1, 1, ref.shape).astype(np.float32) if acc else None
    if acc:
        ref = ref + prev
    ref = np.maximum(ref, 0)
    wb = torch.empty(B.small_conv_weight_elems(C, K, F, F), device="cuda")
    B.small_pack_conv_weights(ctx(), dev(w), wb, C, K, F, F)
    OH, OW = ref.shape[2:]
    out = to_blk(prev) if acc else new_blk(N, K, OH, OW)
    with conv_path("cuda_cores"):
        assert B.small_conv2d_path(ctx(), N, C, K, H, W, F, F, S, pad, B.MATH_FP32) == 1
        B.small_conv2d(ctx(), to_blk(x), wb, dev(b), out, N, C, K, H, W, F, F, S, pad, B.RELU | (B.ACCUMULATE if acc else 0))
    assert rel_err(from_blk(out, N, K, OH, OW), ref) <= 1e-5
    assert pad_lanes_are_zero(out, N, K, OH, OW)
    assert B.small_device_status(ctx()) == 0
