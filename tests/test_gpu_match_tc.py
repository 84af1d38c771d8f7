"""The tcgen05 matching kernel at the edges of its tiles (strips of 4 cells, 32 frames, stages of 64 channels, a tile's
channel range in 1 to 8 chunks over as many CTAs), against the CPU oracle; and the same bits whether the chunks of a tile
are summed by one CTA or by several."""
import pytest
import torch

import paper_2605_07355_b200 as P
from tests.parity import check_clip, to_device
from tests.test_gpu_parity import corr_clip

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("r", [0, 1, 2])
@pytest.mark.parametrize("shape", [(1, 3, 4, 64), (5, 4, 5, 128), (31, 3, 7, 200), (32, 2, 9, 264), (33, 5, 3, 520), (3, 6, 8, 1032),
                                   (65, 1, 4, 1160), (9, 16, 17, 2056)])
def test_tile_edges(shape, r):
    X = corr_clip(*shape, seed=sum(shape) + r, dtype="bf16")
    check_clip(X, r, 0.6)
    check_clip(X, r, 0.6, anchor_mode=2)


@pytest.mark.parametrize("shape,r,clips", [((6, 8, 8, 1024), 1, 24), ((32, 8, 8, 512), 1, 16), ((9, 7, 6, 576), 0, 32),
                                           ((20, 9, 8, 1160), 2, 12)])
def test_bits_do_not_depend_on_the_split(shape, r, clips):
    """thresholds that are the similarity of some token, bit for bit: the strict gate flips on any difference"""
    X = to_device(corr_clip(*shape, seed=sum(shape), dtype="bf16"))
    q = P.ttf_query(X, r, 0.6)
    sims = torch.sort(q["best_sim"][q["best_sim"] < 1.0]).values
    for t in sims[:: max(1, sims.numel() // 8)].tolist():
        one = P.ttf_compress(X, r, t)
        L = int(one[1])
        for lanes in (0, 8):                                 # groups, and single clips that count with their neighbours
            P.ttf_set_schedule(lanes)
            try:
                toks, cnts, poss = P.ttf_compress_batch([X] * clips, r, t)
            finally:
                P.ttf_set_schedule(0)
            torch.cuda.synchronize()
            assert all(int(c) == L for c in cnts)
            assert all(torch.equal(p[:L], one[2][:L]) for p in poss)


@pytest.mark.parametrize("r", [0, 1, 2])
@pytest.mark.parametrize("shape", [(2, 4, 4, 64), (7, 5, 4, 136), (8, 4, 9, 512), (8, 7, 3, 1032), (9, 6, 5, 264), (15, 1, 6, 200), (16, 2, 8, 520),
                                   (16, 9, 7, 1160), (17, 4, 4, 128), (24, 8, 5, 576), (40, 4, 7, 72), (48, 6, 3, 328)])
def test_tiles_of_fewer_frames(shape, r):
    """tiles of 8 and 16 frames over four and two grid rows: frames, rows and cells that end inside a tile"""
    X = corr_clip(*shape, seed=sum(shape) + r, dtype="bf16")
    check_clip(X, r, 0.6)
    check_clip(X, r, 0.6, anchor_mode=1)


@pytest.mark.parametrize("shape,r,clips", [((6, 8, 8, 1024), 1, 24), ((40, 8, 8, 1024), 1, 24), ((16, 16, 16, 1024), 2, 24)])
def test_bits_of_tiles_of_fewer_frames(shape, r, clips):
    """a tile as a cluster, and as fewer CTAs (the second two, the third one) that sum several chunks each"""
    test_bits_do_not_depend_on_the_split(shape, r, clips)


@pytest.mark.parametrize("C,ctas", [(1024, 8), (512, 4)])
def test_as_many_clusters_as_run_at_once_and_one_more(C, ctas):
    """tiles of one grid row of a clip of 32 frames, as many as run at the same time as clusters of eight and of four CTAs, and one
    more (33 and 34, 71 and 72 of them on 148 SMs): then a tile has half as many, which sum two parts of its channels each"""
    fits = max(n for n in range(1, 2 * 148 // ctas + 1) if P.ttf_debug_match_split(32, 1, 4 * n, C, 1) == (1, ctas, ctas))
    assert P.ttf_debug_match_split(32, 1, 4 * (fits + 1), C, 1) == (1, ctas, ctas // 2)      # (not fewer parts: fewer CTAs)
    for tiles in (fits, fits + 1):
        shape = (32, 1, 4 * tiles, C)
        check_clip(corr_clip(*shape, seed=tiles, dtype="bf16"), 1, 0.6)
        test_bits_do_not_depend_on_the_split(shape, 1, 24)


@pytest.mark.parametrize("shape", [(8, 8, 8, 4096), (4, 12, 12, 4096), (8, 10, 10, 4096)])
def test_error_of_the_similarities_of_short_clips(shape):
    """Against 64 bits.  A sum in tensor memory loses at most 2^-23 of its value per addition, half of that on average, and half of
    it again while it grows: n additions n 2^-25.  Eight parts of 4096 channels are 32 additions of 16 channels each."""
    F, H, W, C = shape
    X = to_device(corr_clip(*shape, seed=sum(shape), dtype="bf16"))
    q = P.ttf_query(X, 1, 0.6)
    x = X.double()
    x = x / x.norm(dim=-1, keepdim=True)
    anchor = x[int(q["anchor"])]
    best = torch.full((F, H, W), -2.0, dtype=torch.float64, device="cuda")
    for dy in (-1, 0, 1):
        for dx in (-1, 0, 1):
            y0, y1, x0, x1 = max(0, -dy), min(H, H - dy), max(0, -dx), min(W, W - dx)
            sim = (x[:, y0:y1, x0:x1] * anchor[y0 + dy:y1 + dy, x0 + dx:x1 + dx]).sum(-1)
            best[:, y0:y1, x0:x1] = torch.maximum(best[:, y0:y1, x0:x1], sim)
    best[int(q["anchor"])] = 1.0
    assert float((q["best_sim"].view(F, H, W).double() - best).norm() / best.norm()) < 32 * 2.0 ** -25


def test_a_cta_never_sums_more_parts_than_its_tensor_memory_holds():
    """so many tiles that one CTA each would fill the GPU, in eight parts of 48 columns"""
    shape, clips = (8, 20, 8, 1024), 32
    assert P.ttf_debug_match_split(*shape, 1, clips=16, lanes=2) == (4, 8, 2) and P.ttf_debug_match_split(*shape, 1) == (4, 8, 8)
    test_bits_do_not_depend_on_the_split(shape, 1, clips)


@pytest.mark.parametrize("shape,r,clips,group", [((40, 16, 16, 1024), 1, 16, (8, 2)), ((23, 24, 23, 520), 1, 8, (4, 2)),
                                                 ((17, 21, 11, 1496), 0, 16, (8, 2)), ((24, 20, 15, 248), 1, 3, (3, 1))])
def test_bits_do_not_depend_on_the_tile(shape, r, clips, group):
    """clips whose tile alone has other rows than in a group of the batch"""
    alone = P.ttf_debug_match_split(*shape, r)
    grouped = P.ttf_debug_match_split(*shape, r, *group)
    assert alone[0] != grouped[0] and alone[1] == grouped[1]
    test_bits_do_not_depend_on_the_split(shape, r, clips)
