"""The gather against the CPU oracle where its windows, batches and pieces end: clips of exactly one window of flags, one
token more, several windows, more frames than a warp scans; rows from 16 bytes (32 per batch) to more than a slot."""
import pytest
import torch

import paper_2605_07355_b200 as P
from tests.parity import check_clip, to_device
from tests.test_gpu_parity import corr_clip

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(64, 16, 16, 8), (31, 23, 23, 8), (5, 57, 61, 8), (40, 32, 32, 16), (1100, 4, 4, 8),
                                   (2, 129, 127, 8), (3, 5, 7, 4096), (3, 5, 7, 4104), (2, 3, 3, 12296), (9, 8, 8, 2048),
                                   (7, 9, 11, 1032)])
@pytest.mark.parametrize("kw", [dict(), dict(anchor_mode=2, order=1, pos_base=7)])
def test_windows_and_batches(shape, kw):
    X = corr_clip(*shape, seed=sum(shape), dtype="bf16", sigma=0.6)
    for t in (-2.0, 0.6, 2.0):                               # only the anchor block, a mixture, every token
        check_clip(X, 1, t, **kw)


@pytest.mark.parametrize("shape", [(6, 5, 7, 64), (70, 16, 16, 8)])
def test_segment_has_no_anchor_block(shape):
    X = to_device(corr_clip(*shape, seed=5, dtype="bf16", sigma=0.6))
    N = shape[1] * shape[2]
    full, cnt, pos = P.ttf_compress(X, 1, 0.6, anchor_mode=1)
    for _ in range(2):
        seg, scnt, spos = P.ttf_compress_segment(X, 1, 0.6, frame_base=11)
    n = int(scnt)
    assert n == int(cnt) - N and n > 0
    assert torch.equal(seg[:n], full[N:N + n])
    assert torch.equal(spos[:n], pos[N:N + n] + torch.tensor([10, 0, 0], dtype=torch.int32, device="cuda"))


@pytest.mark.parametrize("shape,dtype", [((2, 2, 3, 4096), "bf16"), ((3, 3, 4, 4104), "bf16"), ((5, 4, 5, 6152), "bf16"),      # 1, 2, 2 pieces
                                         ((4, 3, 3, 2052), "f32"), ((3, 2, 2, 8200), "bf16"),                                   # 2, 3 pieces
                                         ((70, 16, 15, 2056), "bf16"), ((33, 23, 22, 4104), "bf16"),                            # several windows
                                         ((40, 3, 4, 64), "bf16"), ((40, 3, 4, 72), "bf16"), ((260, 9, 8, 16), "f32"),          # 128, 144, 64 bytes
                                         ((1030, 2, 2, 4104), "bf16"), ((1, 1, 1, 4104), "bf16")])
def test_rows_of_pieces_and_rows_that_fill_no_slot(shape, dtype):
    """alone: a row of up to three pieces of a slot; windows; the smallest rows; more frames than the shared prefix holds"""
    X = corr_clip(*shape, seed=sum(shape), dtype=dtype)
    check_clip(X, 1, 0.6)
    check_clip(X, 1, 0.6, anchor_mode=2, order=1, pos_base=7)
