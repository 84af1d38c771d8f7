"""The frame sums behind the anchor at the slice widths the sweep chooses from (a whole, half and quarter warp across a row),
with channels that do not fill a slice and tokens that do not fill a batch: anchor and everything after it against the CPU
oracle, alone and in a launch over several clips."""
import pytest
import torch

import paper_2605_07355_b200 as P
from tests.parity import check_clip, to_device
from tests.test_gpu_batch import assert_same_as_single
from tests.test_gpu_parity import corr_clip

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape,dtype", [((2, 9, 9, 72), "bf16"), ((3, 17, 31, 200), "bf16"), ((40, 3, 5, 1032), "bf16"),
                                         ((150, 2, 3, 520), "bf16"), ((3, 17, 31, 36), "f32"), ((40, 3, 5, 516), "f32"),
                                         ((150, 2, 3, 260), "f32")])
def test_slice_widths(shape, dtype):
    X = corr_clip(*shape, seed=sum(shape), dtype=dtype)
    check_clip(X, 1, 0.6)
    Xs = [to_device(corr_clip(*shape, seed=sum(shape) + j, dtype=dtype)) for j in range(6)]
    outs = P.ttf_compress_batch(Xs, 1, 0.6)
    torch.cuda.synchronize()
    assert_same_as_single(Xs, 1, 0.6, outs)
