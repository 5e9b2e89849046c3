"""The quantised convolution's tilings at their edges, bit-exact against the oracle: column tiles of wide planes, filter tiles
with a remainder, filters that stream instead of staying resident, several images per tile, windows whose border classes
are too many for the table, windows taller than one input box, more filter tiles than the chip has SMs, and every form of the
requantising shift."""
import numpy as np
import pytest
import torch

import oracle
from paper_2303_04769_b200 import binding as B
from gpu_util import ctx
from test_gpu_quant import dev, multiplier, pad_lanes_zero, q_blk, q_nchw, u8

pytestmark = pytest.mark.gpu

CASES = [  # N, C, K, H, W, FH, FW, S, pad, shift
    (1, 40, 33, 3, 300, 3, 3, 1, (1, 1, 1, 1), 40),      # rows wider than a box: column tiles
    (1, 40, 20, 9, 301, 3, 3, 2, (1, 1, 1, 1), 36),      # the same over phase planes
    (2, 33, 160, 12, 13, 3, 3, 1, (1, 1, 1, 1), 43),     # two filter tiles, the second one ragged
    (3, 600, 64, 6, 6, 3, 3, 1, (1, 1, 1, 1), 44),       # more filters than shared memory holds: streamed
    (150, 96, 128, 7, 7, 3, 3, 1, (1, 1, 1, 1), 38),     # several images per tile, the last tile ragged
    (2, 32, 24, 17, 31, 1, 1, 1, (0, 0, 0, 0), 31),      # pointwise, 527 pixels per plane
    (1, 8, 40, 25, 12, 9, 3, 1, (8, 8, 2, 2), 33),       # 729 border classes
    (1, 4, 8, 200, 5, 180, 1, 1, (3, 0, 0, 0), 40),      # a tall window
    (1, 4, 8, 256, 3, 256, 1, 2, (1, 0, 0, 0), 41),      # the tallest, over phase planes: two boxes per strip
    (2, 5, 18977, 12, 11, 3, 3, 1, (1, 1, 1, 1), 39),    # more filter tiles than SMs
    (3, 33, 37900, 7, 5, 1, 1, 2, (0, 0, 0, 0), 36),     # more than two per SM, the last one ragged
]


@pytest.mark.parametrize("case", CASES)
def test_q_conv_tilings_bit_exact(case):
    N, C, K, H, W, FH, FW, S, pad, shift = case
    x, w = u8((N, C, H, W), 21), u8((K, C, FH, FW), 22)
    b = np.random.RandomState(23).randint(-9000, 9000, size=K).astype(np.int32)
    zx, zw, zo = 117, 131, 60
    mult, shift = multiplier(C * FH * FW, zx, zw, shift)
    wb = torch.full((B.small_q_conv_weight_bytes(C, K, FH, FW),), 0x5A, dtype=torch.uint8, device="cuda")
    B.small_q_pack_conv_weights(ctx(), dev(w), wb, C, K, FH, FW)
    ref = oracle.q_conv2d(x, w, b, S, pad, zx, zw, zo, mult, shift, False)
    OH, OW = ref.shape[2:]
    out = torch.full((B.small_q_packed_bytes(N, K, OH, OW),), 0xEE, dtype=torch.uint8, device="cuda")
    B.small_q_conv2d(ctx(), q_blk(x), wb, dev(b), out, N, C, K, H, W, FH, FW, S, pad, (zx, zw, zo, mult, shift), 0)
    got = q_nchw(out, N, K, OH, OW)
    assert B.small_device_status(ctx()) == 0
    assert len(np.unique(ref)) > 3
    np.testing.assert_array_equal(got, ref)
    assert pad_lanes_zero(out, N, K, OH, OW)


@pytest.mark.parametrize("case", [(1, 40, 5, 7, 1, 29), (3, 16, 33, 6, 1, 43), (2, 70, 12, 12, 2, 44), (40, 64, 25, 5, 1, 36), (2, 8, 3, 3, 2, 36)])
def test_q_depthwise_3x3_runs_bit_exact(case):
    """Runs of rows of every length (ragged last run, fewer rows than a trip), both strides, every form of the shift."""
    N, C, H, W, S, shift = case
    x, w = u8((N, C, H, W), 24), u8((C, 3, 3), 25)
    b = np.random.RandomState(26).randint(-3000, 3000, size=C).astype(np.int32)
    mult, shift = multiplier(9, 120, 131, shift)
    wb = torch.empty(B.small_q_dw_weight_bytes(C, 3, 3), dtype=torch.uint8, device="cuda")
    B.small_q_pack_dw_weights(ctx(), dev(w), wb, C, 3, 3)
    ref = oracle.q_dwconv2d(x, w, b, S, (1, 1, 1, 1), 120, 131, 70, mult, shift, True)
    OH, OW = ref.shape[2:]
    out = torch.full((B.small_q_packed_bytes(N, C, OH, OW),), 0xEE, dtype=torch.uint8, device="cuda")
    B.small_q_dwconv2d(ctx(), q_blk(x), wb, dev(b), out, N, C, H, W, 3, 3, S, (1, 1, 1, 1), (120, 131, 70, mult, shift), B.RELU)
    np.testing.assert_array_equal(q_nchw(out, N, C, OH, OW), ref)
    assert pad_lanes_zero(out, N, C, OH, OW)
