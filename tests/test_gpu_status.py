"""The give-up path of the bounded device waits, driven without a fault or a hang: a test hook makes every copy
barrier expect 16 bytes more than its copy delivers and lowers the poll limit, so the data lands, the barrier never
completes, the waiting lane runs out of polls, stops and sets the error word."""
import numpy as np
import pytest
import torch

import paper_2605_07355_b200 as P
from paper_2605_07355_b200 import binding as B
from tests.parity import check_clip, to_device
from tests.test_gpu_parity import corr_clip

pytestmark = pytest.mark.gpu


def test_copy_wait_runs_out_then_the_next_call_is_clean():
    X = corr_clip(6, 6, 7, 256, seed=77, dtype="bf16")
    Xd = to_device(X)
    st = torch.cuda.Stream()
    ref = P.ttf_compress(Xd, 1, 0.7, stream=st)
    assert P.ttf_last_device_status(st) == B.TTF_OK
    L = int(ref[1].item())
    assert L > 6 * 7
    P.ttf_debug_set_wait(32, 16)
    try:
        toks, cnt, pos = P.ttf_compress(Xd, 1, 0.7, stream=st)
        assert P.ttf_last_device_status(st) == B.TTF_ERR_TIMEOUT        # synchronises the stream
        assert int(cnt.item()) == -1
        # a batch reports through the caller's stream
        outs = P.ttf_compress_batch([Xd, Xd, Xd], 1, 0.7, stream=st)
        assert P.ttf_last_device_status(st) == B.TTF_ERR_TIMEOUT
        assert all(int(c.item()) == -1 for c in outs[1])
    finally:
        P.ttf_debug_set_wait()
    # the same stream, hence the same scratch block: nothing of the failed calls is left
    toks, cnt, pos = P.ttf_compress(Xd, 1, 0.7, stream=st)
    assert P.ttf_last_device_status(st) == B.TTF_OK
    assert int(cnt.item()) == L
    assert torch.equal(toks[:L], ref[0][:L]) and torch.equal(pos[:L], ref[2][:L])
    outs = P.ttf_compress_batch([Xd, Xd, Xd], 1, 0.7, stream=st)
    assert P.ttf_last_device_status(st) == B.TTF_OK
    assert all(int(c.item()) == L for c in outs[1])
    with torch.cuda.stream(st):
        check_clip(X, 1, 0.7, stream=st)                                 # and it still equals the oracle


@pytest.mark.parametrize("C", [64, 256, 2048])
def test_tensor_core_pipeline_gives_up_and_recovers(C):
    """the tcgen05 matching kernel under the same hook: its copy barriers never complete, so its MMA issuer, its
    epilogue warps and then its producer run out of polls; the CTAs (alone for C = 64, in clusters of 2 for C = 256
    and of 8 for C = 2048) still meet at their barriers, free their tensor memory and return; the query reports the time-out
    and the next call is clean"""
    X = corr_clip(6, 6, 7, C, seed=79, dtype="bf16")
    Xd = to_device(X)
    st = torch.cuda.Stream()
    P.ttf_set_match_kernel(2)
    try:
        ref = P.ttf_query(Xd, 1, 0.7, stream=st)
        assert P.ttf_last_device_status(st) == B.TTF_OK
        P.ttf_debug_set_wait(32, 16)
        try:
            P.ttf_query(Xd, 1, 0.7, stream=st)
            assert P.ttf_last_device_status(st) == B.TTF_ERR_TIMEOUT
            _, cnt, _ = P.ttf_compress(Xd, 1, 0.7, stream=st)
            assert P.ttf_last_device_status(st) == B.TTF_ERR_TIMEOUT and int(cnt.item()) == -1
        finally:
            P.ttf_debug_set_wait()
        again = P.ttf_query(Xd, 1, 0.7, stream=st)
        assert P.ttf_last_device_status(st) == B.TTF_OK
        for k in ref:
            assert torch.equal(ref[k], again[k]), k
        with torch.cuda.stream(st):
            check_clip(X, 1, 0.7, stream=st)
    finally:
        P.ttf_set_match_kernel(0)


@pytest.mark.parametrize("r,clips", [(1, 24), (2, 24)])
def test_tiles_of_one_cta_and_several_chunks_give_up_and_recover(r, clips):
    """large launches: every tile is one CTA that sums all chunks of its channels (8 alone, 4 for r = 2) itself"""
    X = corr_clip(32, 8, 8, 1024, seed=82, dtype="bf16")
    assert P.ttf_debug_match_split(*X.shape, r, clips=clips // 2, lanes=2) == (1, 4 if r == 2 else 8, 1)
    Xs = [to_device(X)] * clips
    st = torch.cuda.Stream()
    ref = P.ttf_compress(Xs[0], r, 0.7, stream=st)
    L = int(ref[1].item())
    P.ttf_compress_batch(Xs, r, 0.7, stream=st)
    assert P.ttf_last_device_status(st) == B.TTF_OK
    P.ttf_debug_set_wait(32, 16)
    try:
        _, cnts, _ = P.ttf_compress_batch(Xs, r, 0.7, stream=st)
        assert P.ttf_last_device_status(st) == B.TTF_ERR_TIMEOUT
        assert all(int(c) == -1 for c in cnts)
    finally:
        P.ttf_debug_set_wait()
    toks, cnts, poss = P.ttf_compress_batch(Xs, r, 0.7, stream=st)
    assert P.ttf_last_device_status(st) == B.TTF_OK
    for t, c, p in zip(toks, cnts, poss):
        assert int(c) == L and torch.equal(t[:L], ref[0][:L]) and torch.equal(p[:L], ref[2][:L])


def test_status_of_caller_owned_and_built_in_scratch():
    X = corr_clip(4, 5, 5, 128, seed=78, dtype="bf16")
    Xd = to_device(X)
    nbytes = P.ttf_workspace_bytes(4, 5, 5, 128, 1, 1)
    ws = torch.empty(nbytes, dtype=torch.uint8, device="cuda")
    P.ttf_debug_set_wait(32, 16)
    try:
        _, cnt, _ = P.ttf_compress(Xd, 1, 0.7, workspace=ws)
        assert P.ttf_workspace_status(ws) == B.TTF_ERR_TIMEOUT and int(cnt.item()) == -1
    finally:
        P.ttf_debug_set_wait()
    _, cnt, _ = P.ttf_compress(Xd, 1, 0.7, workspace=ws)
    assert P.ttf_workspace_status(ws) == B.TTF_OK and int(cnt.item()) > 0
    out = {"keep": torch.empty(100, dtype=torch.uint8, device="cuda")}
    P.ttf_query_static(Xd, 1, 0.7, out)
    assert P.ttf_workspace_status(None) == B.TTF_OK
    assert P.ttf_last_device_status(torch.cuda.Stream()) == B.TTF_OK      # a stream the library has never seen


def test_a_batch_reports_a_clip_whose_scratch_block_a_later_clip_used():
    """one lane, five clips on two scratch blocks in turn: the first gives up, the others, 2 bytes off a 16-byte boundary,
    take the kernels without bounded waits and come out right"""
    F, H, W, C = 4, 5, 5, 64
    X = corr_clip(F, H, W, C, seed=81, dtype="bf16")
    Xs = [to_device(X)]
    for _ in range(4):
        buf = torch.zeros(X.size + 8, dtype=torch.bfloat16, device="cuda")
        Xs.append(buf[1:1 + X.size].view(F, H, W, C))
        Xs[-1].copy_(Xs[0])
    L = int(P.ttf_compress(Xs[0], 1, 0.7)[1])
    st = torch.cuda.Stream()
    P.ttf_set_schedule(1)
    try:
        P.ttf_compress_batch(Xs, 1, 0.7, stream=st)
        assert P.ttf_last_device_status(st) == B.TTF_OK
        P.ttf_debug_set_wait(32, 16)
        try:
            _, cnts, _ = P.ttf_compress_batch(Xs, 1, 0.7, stream=st)
            assert P.ttf_last_device_status(st) == B.TTF_ERR_TIMEOUT
            assert [int(c) for c in cnts] == [-1] + [L] * 4
        finally:
            P.ttf_debug_set_wait()
        _, cnts, _ = P.ttf_compress_batch(Xs, 1, 0.7, stream=st)
        assert P.ttf_last_device_status(st) == B.TTF_OK and [int(c) for c in cnts] == [L] * 5
        P.ttf_compress(Xs[0], 1, 0.7, stream=st)
        assert P.ttf_last_device_status(st) == B.TTF_OK
    finally:
        P.ttf_set_schedule(0)


def test_the_status_of_a_batch_outlives_its_scratch():
    """a batch over the lanes; then a larger clip on another stream takes the place of the lanes' scratch"""
    Xs = [to_device(corr_clip(4, 5, 5, 64, seed=83, dtype="bf16"))] * 3
    larger = [to_device(corr_clip(40, 16, 16, 512, seed=84, dtype="bf16"))] * 3
    a, b = torch.cuda.Stream(), torch.cuda.Stream()
    P.ttf_release()
    P.ttf_set_schedule(2)
    try:
        for limits, status in (((32, 16), B.TTF_ERR_TIMEOUT), ((), B.TTF_OK)):
            P.ttf_debug_set_wait(*limits)
            P.ttf_compress_batch(Xs, 1, 0.7, stream=a)
            P.ttf_debug_set_wait()
            P.ttf_compress_batch(larger, 1, 0.7, stream=b)
            assert P.ttf_last_device_status(b) == B.TTF_OK
            assert P.ttf_last_device_status(a) == status
            P.ttf_release()
    finally:
        P.ttf_debug_set_wait()
        P.ttf_set_schedule(0)


def test_status_after_a_batch_that_found_no_memory():
    """small batches on the caller's stream: the block of the first makes room for a larger clip's, for which there is no memory"""
    Xs = [to_device(corr_clip(4, 5, 5, 64, seed=85, dtype="bf16"))] * 3
    larger = [to_device(corr_clip(256, 1, 1, 32768, seed=86, dtype="bf16"))] * 3      # (more than 40 MB of scratch each)
    outs = P.ttf_compress_batch(larger, 1, 0.7)              # (loads the kernels, before memory is short)
    torch.cuda.synchronize()
    st = torch.cuda.Stream()
    P.ttf_release()
    P.ttf_debug_set_wait(32, 16)
    try:
        P.ttf_compress_batch(Xs, 1, 0.7, stream=st)
        torch.cuda.synchronize()
    finally:
        P.ttf_debug_set_wait()
    hold, size = [], 64 << 30
    while size >= 16 << 20:
        try:
            hold.append(torch.empty(size, dtype=torch.uint8, device="cuda"))
        except torch.cuda.OutOfMemoryError:
            size //= 2
    try:
        with pytest.raises(P.TTFError):
            P.ttf_compress_batch(larger, 1, 0.7, *outs, stream=st)
        assert P.ttf_last_device_status(st) == B.TTF_ERR_TIMEOUT          # (of the batch before: nothing of the other one ran)
    finally:
        hold.clear()
        torch.cuda.empty_cache()
    P.ttf_compress_batch(larger, 1, 0.7, *outs, stream=st)
    assert P.ttf_last_device_status(st) == B.TTF_OK
