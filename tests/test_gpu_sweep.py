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


@pytest.mark.parametrize("shape,dtype", [((64, 3, 3, 136), "bf16"), ((65, 3, 3, 136), "bf16"), ((32, 3, 4, 264), "bf16"), ((33, 3, 4, 512), "bf16"),
                                         ((7, 4, 4, 512), "bf16"), ((8, 4, 4, 520), "bf16"), ((64, 2, 3, 256), "f32"), ((33, 2, 3, 388), "f32"),
                                         ((9, 3, 3, 2056), "bf16"), ((40, 3, 3, 4096), "bf16")])
def test_statistics_in_one_cta_and_in_a_cluster(shape, dtype):
    """two to four slices of channels at the frames that one CTA holds and one more; frames that leave warps without any"""
    test_slice_widths(shape, dtype)
