"""Max pooling with a 3x3 window, whose taps outside the plane are replaced by taps inside it: values and indices (ties keep
the first position) bit-exact at every border, with padding up to two, strides 1 to 3."""
import numpy as np
import pytest
import torch

import oracle
import synth
from paper_2303_04769_b200 import binding as B
from gpu_util import ctx, to_blk, from_blk, new_blk, pad_lanes_are_zero

pytestmark = pytest.mark.gpu

CASES = [(1, 3, 1, 1, 1, (2, 2, 2, 2)), (2, 33, 5, 4, 1, (2, 1, 0, 2)), (2, 40, 9, 8, 2, (1, 1, 1, 1)), (3, 8, 7, 10, 3, (0, 2, 2, 0)), (1, 64, 28, 27, 2, (0, 1, 0, 1))]


@pytest.mark.parametrize("case", CASES)
def test_max_pool_3x3(case):
    N, C, H, W, S, pad = case
    x = np.round(synth.uniform((N, C, H, W), -2, 2, 9, seed=3)).astype(np.float32)      # many ties
    ref, ref_idx = oracle.pool2d(x, 3, 3, S, pad, "max", with_indices=True)
    OH, OW = ref.shape[2:]
    out, idx = new_blk(N, C, OH, OW), torch.zeros(B.small_packed_elems(N, C, OH, OW), dtype=torch.int32, device="cuda")
    B.small_pool2d(ctx(), to_blk(x), out, idx, N, C, H, W, 3, 3, S, pad, B.POOL_MAX)
    np.testing.assert_array_equal(from_blk(out, N, C, OH, OW), ref)
    got = from_blk(idx.view(torch.float32), N, C, OH, OW).view(np.int32)
    np.testing.assert_array_equal(got, ref_idx)
    assert pad_lanes_are_zero(out, N, C, OH, OW)
    B.small_pool2d(ctx(), to_blk(x), out, None, N, C, H, W, 3, 3, S, pad, B.POOL_MAX)
    np.testing.assert_array_equal(from_blk(out, N, C, OH, OW), ref)
