"""The tiled fp32 matching kernel against the CPU oracle at the edges of its tiles: 8 / 4 frames per warp, up to 32 per
CTA, stages of 128 channels in a ring of 4 / 3, window rows outside the grid."""
import pytest

import paper_2605_07355_b200 as P
from paper_2605_07355_b200 import binding as B
from tests.parity import check_clip, to_device
from tests.test_gpu_parity import corr_clip

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("r", [0, 1, 2])
@pytest.mark.parametrize("shape", [(1, 3, 4, 4), (7, 1, 9, 124), (8, 9, 1, 128), (9, 5, 3, 132), (31, 2, 2, 516),
                                   (33, 4, 5, 640), (65, 3, 3, 260), (34, 16, 17, 64)])
def test_tile_edges(shape, r):
    F, H, W, C = shape
    X = corr_clip(F, H, W, C, seed=sum(shape) + r)
    check_clip(X, r, 0.6)
    check_clip(X, r, 0.6, anchor_mode=2)


def test_gives_up_and_recovers():
    X = corr_clip(9, 5, 6, 1028, seed=80)                    # nine stages: more than the ring holds
    Xd = to_device(X)
    P.ttf_query(Xd, 1, 0.7)
    P.ttf_debug_set_wait(32, 16)
    try:
        P.ttf_query(Xd, 1, 0.7)
        assert P.ttf_last_device_status() == B.TTF_ERR_TIMEOUT
    finally:
        P.ttf_debug_set_wait()
    check_clip(X, 1, 0.7)
    assert P.ttf_last_device_status() == B.TTF_OK


@pytest.mark.parametrize("r", [0, 1, 2])
@pytest.mark.parametrize("shape", [(33, 20, 20, 100), (40, 21, 20, 132), (64, 20, 16, 260), (33, 24, 25, 384), (70, 24, 24, 516)])
def test_rings_of_fewer_stages(shape, r):
    """more units than fit the GPU with the whole ring, rows of one to five stages"""
    check_clip(corr_clip(*shape, seed=sum(shape) + r, dtype="f32"), r, 0.6)
