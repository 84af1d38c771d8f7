"""Launches that cover several clips: every clip of a batch gives what the call for that clip alone gives, for batches
that fill one group, leave the last one ragged, or take several turns per lane, through every matching kernel."""
import pytest
import torch

import paper_2605_07355_b200 as P
from tests.parity import to_device
from tests.test_gpu_batch import assert_same_as_single
from tests.test_gpu_parity import corr_clip

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("clips", [2, 3, 33, 81])            # groups of 1 + 1, 2 + 1, 16 + 16 + 1, five of 16 + 1
@pytest.mark.parametrize("shape,dtype,r", [((5, 4, 6, 64), "bf16", 1), ((3, 5, 4, 128), "bf16", 2), ((4, 3, 5, 36), "f32", 1),
                                           ((3, 4, 4, 33), "bf16", 1), ((2, 3, 3, 8), "f32", 3), ((130, 2, 2, 4100), "bf16", 1)])
def test_groups_match_single_calls(shape, dtype, r, clips):
    if shape[0] > 100 and clips > 3:
        clips = 3                                            # (frames and channels beyond the statistics cluster)
    Xs = [to_device(corr_clip(*shape, seed=500 + j, dtype=dtype)) for j in range(min(clips, 9))]
    Xs = [Xs[j % len(Xs)] for j in range(clips)]
    for rep in range(2):
        outs = P.ttf_compress_batch(Xs, r, 0.6)
    torch.cuda.synchronize()
    assert P.ttf_last_device_status() == 0
    assert_same_as_single(Xs, r, 0.6, outs)


def test_clips_of_different_alignment():
    F, H, W, C = 3, 4, 5, 64
    Xs = []
    for j in range(4):
        buf = torch.zeros(F * H * W * C + 8, dtype=torch.bfloat16, device="cuda")
        view = buf[j % 2:j % 2 + F * H * W * C].view(F, H, W, C)          # every second clip 2 bytes off
        view.copy_(to_device(corr_clip(F, H, W, C, seed=600 + j, dtype="bf16")))
        Xs.append(view)
    outs = P.ttf_compress_batch(Xs, 1, 0.6)
    torch.cuda.synchronize()
    assert_same_as_single(Xs, 1, 0.6, outs)
