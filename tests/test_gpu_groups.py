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


def test_outputs_of_different_alignment():
    """21 clips, the token rows of every third 2 bytes off"""
    Xs = [to_device(corr_clip(3, 4, 5, 64, seed=620 + j, dtype="bf16")) for j in range(21)]
    toks, cnts, poss = outputs(Xs[0], 21)
    for j in range(0, 21, 3):
        toks[j] = torch.zeros(toks[j].numel() + 8, dtype=toks[j].dtype, device="cuda")[1:1 + toks[j].numel()].view(toks[j].shape)
    assert_same_as_single(Xs, 1, 0.6, P.ttf_compress_batch(Xs, 1, 0.6, toks, cnts, poss))


def outputs(X, n):
    rows, C = X.shape[0] * X.shape[1] * X.shape[2], X.shape[3]
    return ([torch.zeros((rows, C), dtype=X.dtype, device="cuda") for _ in range(n)],
            [torch.zeros(1, dtype=torch.int32, device="cuda") for _ in range(n)],
            [torch.zeros((rows, 3), dtype=torch.int32, device="cuda") for _ in range(n)])


def captured(Xs, outs, st):
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=st):
        P.ttf_compress_batch(Xs, 1, 0.6, *outs, stream=st)
    return g


def assert_replays(g, Xs, outs):
    for c in outs[1]:
        c.zero_()
    g.replay()
    torch.cuda.synchronize()
    assert_same_as_single(Xs, 1, 0.6, outs)


def test_scratch_and_captures_after_eight_clips():
    """batches of up to 16 clips take no more device memory than the one of eight, and a capture, which cannot allocate, takes
    any number of clips"""
    Xs = [to_device(corr_clip(16, 32, 32, 64, seed=700 + j, dtype="bf16")) for j in range(5)]
    Xs = [Xs[j % 5] for j in range(33)]
    outs = outputs(Xs[0], 33)
    P.ttf_release()
    assert_same_as_single(Xs[:8], 1, 0.6, P.ttf_compress_batch(Xs[:8], 1, 0.6))      # (loads the kernels for one clip, too)
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    for n in (9, 16):
        P.ttf_compress_batch(Xs[:n], 1, 0.6, *[o[:n] for o in outs])
    torch.cuda.synchronize()
    assert torch.cuda.mem_get_info()[0] == before
    st = torch.cuda.Stream()
    assert_replays(captured(Xs, outs, st), Xs, outs)
    P.ttf_release()
    P.ttf_compress_batch(Xs[:2], 1, 0.6)                     # one block per lane: single clips, one after the other
    assert_replays(captured(Xs[:7], [o[:7] for o in outs], st), Xs[:7], [o[:7] for o in outs])
    assert_same_as_single(Xs + Xs, 1, 0.6, P.ttf_compress_batch(Xs + Xs, 1, 0.6))    # several turns per lane


def test_graphs_of_smaller_batches_stay_valid():
    """every batch of the row is larger than the one before it; the graphs captured with the smaller ones are replayed after it"""
    Xs = [to_device(corr_clip(4, 16, 16, 64, seed=720 + j, dtype="bf16")) for j in range(5)]
    Xs = [Xs[j % 5] for j in range(20)]
    P.ttf_release()
    st = torch.cuda.Stream()
    graphs = []
    for n in (1, 2, 3, 5, 8, 20):
        outs = outputs(Xs[0], n)
        P.ttf_compress_batch(Xs[:n], 1, 0.6, *outs, stream=st)
        torch.cuda.synchronize()
        for g, m, o in graphs:
            assert_replays(g, Xs[:m], o)
        graphs.append((captured(Xs[:n], outs, st), n, outs))
    for g, m, o in graphs:
        assert_replays(g, Xs[:m], o)


def test_bench_counts_the_launches_of_a_step():
    """each kernel once per group of a batch, once per clip where clips go alone; no statistics for a fixed anchor"""
    from bench import count_launches
    Xs = [to_device(corr_clip(4, 5, 6, 64, seed=740, dtype="bf16"))] * 16
    assert count_launches(lambda: P.ttf_compress_batch(Xs, 1, 0.6)) == 2 * 4
    assert count_launches(lambda: P.ttf_compress_batch(Xs, 1, 0.6, anchor_mode=1)) == 2 * 3
    assert count_launches(lambda: P.ttf_compress(Xs[0], 1, 0.6)) == 4
    P.ttf_set_schedule(3)
    try:
        assert count_launches(lambda: P.ttf_compress_batch(Xs, 1, 0.6)) == 16 * 4
    finally:
        P.ttf_set_schedule(0)
