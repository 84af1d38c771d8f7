"""Batches of few bytes run on the caller's own stream: up to eight clips in one launch of each kernel, up to sixteen in two.
Every clip comes out as from the call for it alone, also where the stream's blocks hold another shape's data, where two
streams work at the same time, where a capture finds no scratch on its stream, and for a stream handle that means another
stream in every thread."""
import ctypes
import threading

import pytest
import torch

import paper_2605_07355_b200 as P
from tests.parity import to_device
from tests.test_gpu_batch import assert_same_as_single
from tests.test_gpu_groups import assert_replays, captured, outputs
from tests.test_gpu_parity import corr_clip

pytestmark = pytest.mark.gpu


def clips_of(shape, n, dtype="bf16", seed=900):
    return [to_device(corr_clip(*shape, seed=seed + j, dtype=dtype)) for j in range(n)]


@pytest.mark.parametrize("n", [1, 2, 7, 8, 9, 15, 16, 17])
@pytest.mark.parametrize("shape,dtype", [((5, 4, 6, 64), "bf16"), ((3, 4, 4, 33), "bf16"), ((4, 3, 5, 36), "f32"),
                                         ((130, 2, 2, 4100), "bf16")])       # (the last: statistics with an arrival counter)
def test_every_clip_as_alone_on_dirty_blocks(shape, dtype, n):
    Xs, other = clips_of(shape, n, dtype), clips_of((7, 6, 9, 200), 3)
    st = torch.cuda.Stream()
    for _ in range(2):
        P.ttf_compress_batch(other, 1, 0.6, stream=st)
        outs = P.ttf_compress_batch(Xs, 1, 0.6, stream=st)
    assert P.ttf_last_device_status(st) == P.TTF_OK
    assert_same_as_single(Xs, 1, 0.6, outs)
    for kw in (dict(anchor_mode=1), dict(anchor_mode=2, order=1, pos_base=3)):
        toks, cnts, poss = P.ttf_compress_batch(Xs, 1, 0.6, stream=st, **kw)
        st.synchronize()
        for X, t, c, p in zip(Xs, toks, cnts, poss):
            a = P.ttf_compress(X, 1, 0.6, **kw)
            L = int(a[1])
            assert int(c) == L and torch.equal(t[:L], a[0][:L]) and torch.equal(p[:L], a[2][:L])


def test_two_streams_and_two_threads():
    """batches on two streams from two threads, each of which also makes single calls on a stream of the two"""
    sets = [clips_of((6, 5, 7, 128), 5, seed=930), clips_of((9, 6, 6, 72), 8, seed=950)]
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    results, alone = {}, {0: [], 1: []}

    def work(i):
        outs = []
        for n in range(20):
            outs += [P.ttf_compress_batch(sets[i], 1, 0.6, stream=st) for st in streams]
            alone[i].append(P.ttf_compress(sets[i][n % 5], 1, 0.6, stream=streams[i]))
        results[i] = outs
    threads = [threading.Thread(target=work, args=(i,)) for i in range(2)]
    [t.start() for t in threads]
    [t.join() for t in threads]
    torch.cuda.synchronize()
    for i in range(2):
        for outs in (results[i][0], results[i][-2], results[i][-1]):
            assert_same_as_single(sets[i], 1, 0.6, outs)
        for n, (tok, cnt, pos) in enumerate(alone[i]):
            ref = results[i][-1]
            L = int(ref[1][n % 5])
            assert int(cnt) == L and torch.equal(tok[:L], ref[0][n % 5][:L]) and torch.equal(pos[:L], ref[2][n % 5][:L])


def test_more_streams_than_hold_scratch():
    """64 streams hold scratch of their own; batches on further ones take the lanes, and after ttf_release theirs again"""
    Xs = clips_of((5, 4, 6, 64), 3, seed=910)
    streams = []
    try:
        for _ in range(66):
            h = ctypes.c_void_p()
            assert int(torch.cuda.cudart().cudaStreamCreate(ctypes.addressof(h))) == 0
            streams.append(h.value)
        P.ttf_release()
        for _ in range(2):
            outs = [P.ttf_compress_batch(Xs, 1, 0.6, stream=st) for st in streams]
            torch.cuda.synchronize()
            for o in outs[:2] + outs[-4:]:
                assert_same_as_single(Xs, 1, 0.6, o)
            assert P.ttf_last_device_status(streams[-1]) == P.TTF_OK
        P.ttf_release()
        assert_same_as_single(Xs, 1, 0.6, P.ttf_compress_batch(Xs, 1, 0.6, stream=streams[-1]))
    finally:
        torch.cuda.synchronize()
        P.ttf_release()
        for st in streams:
            torch.cuda.cudart().cudaStreamDestroy(st)


def test_capture_on_a_stream_without_scratch_and_with_it():
    Xs = clips_of((6, 5, 7, 128), 8, seed=970)
    P.ttf_release()
    P.ttf_compress_batch(clips_of((64, 16, 16, 1024), 8), 1, 0.6)   # (128 MB and more: over the lanes, which now hold scratch)
    for n in (3, 8):
        st = torch.cuda.Stream()
        outs = outputs(Xs[0], n)
        first = captured(Xs[:n], outs, st)
        assert_replays(first, Xs[:n], outs)
        P.ttf_compress_batch(Xs[:n], 1, 0.6, *outs, stream=st)
        torch.cuda.synchronize()
        second = captured(Xs[:n], outs, st)
        for g in (first, second, first):
            assert_replays(g, Xs[:n], outs)


def test_per_thread_default_stream():
    Xs = clips_of((6, 5, 7, 128), 4, seed=990)
    torch.cuda.synchronize()
    outs = outputs(Xs[0], 4)
    torch.cuda.synchronize()
    P.ttf_compress_batch(Xs, 1, 0.6, *outs, stream=2)               # cudaStreamPerThread
    torch.cuda.synchronize()
    assert_same_as_single(Xs, 1, 0.6, outs)


@pytest.mark.parametrize("dtype,r,n,channels,launches", [("bf16", 1, 12, 64, 2), ("bf16", 2, 12, 1024, 2), ("f32", 2, 9, 264, 2), ("bf16", 1, 5, 1024, 1),
                                                         ("bf16", 1, 5, 8192, 2), ("f32", 3, 9, 64, 2)])
def test_every_clip_as_alone_on_both_sides_of_the_line(dtype, r, n, channels, launches):
    """batches of 9 to 16 clips that take the caller's stream or the lanes by what their matching costs, and of five below and above
    45 MB: one launch of each kernel or two"""
    from bench import count_launches
    Xs = clips_of((8, 9, 8, channels), 3, dtype, seed=1010)
    Xs = [Xs[j % 3] for j in range(n)]
    if channels == 8192:
        Xs = clips_of((60, 4, 3, channels), 3, dtype, seed=1020)
        Xs = [Xs[j % 3] for j in range(n)]
    outs = P.ttf_compress_batch(Xs, r, 0.6)
    assert P.ttf_last_device_status() == P.TTF_OK
    assert_same_as_single(Xs, r, 0.6, outs)
    assert count_launches(lambda: P.ttf_compress_batch(Xs, r, 0.6)) == launches * 4
