"""A fixed anchor on a clip of one window of flags: the matching kernel is the first kernel of the call.  Results against the
CPU oracle on scratch that other shapes and calls have used, at the edges of the rule, and the report of a wait that ran out,
of this call and not of the next."""
import pytest
import torch

import paper_2605_07355_b200 as P
from paper_2605_07355_b200 import binding as B
from tests.parity import check_clip, to_device
from tests.test_gpu_parity import corr_clip

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape,dtype", [((1, 2, 3, 64), "bf16"), ((6, 5, 7, 200), "bf16"), ((9, 8, 8, 72), "f32"), ((64, 16, 16, 64), "bf16"),
                                         ((16, 32, 33, 64), "bf16"), ((5, 4, 6, 32), "bf16"), ((4, 3, 5, 33), "bf16"),
                                         ((1026, 2, 2, 64), "bf16"), ((7, 4, 4, 2056), "f32")])
def test_between_calls_of_other_kinds(shape, dtype):
    X, other = corr_clip(*shape, seed=sum(shape), dtype=dtype), to_device(corr_clip(12, 9, 7, 264, seed=3, dtype="bf16"))
    for kw in (dict(anchor_mode=1), dict(anchor_mode=2, order=1, pos_base=5), dict(anchor_mode=3, anchor_frame=shape[0] // 2)):
        P.ttf_compress(other, 1, 0.6)
        check_clip(X, 1, 0.6, **kw)
        P.ttf_query(other, 1, 0.6, anchor_mode=2)
        check_clip(X, 1, 0.6, **kw)
    seg = P.ttf_compress_segment(to_device(X), 1, 0.6, frame_base=3)
    full = P.ttf_compress(to_device(X), 1, 0.6, anchor_mode=1)
    N, n = shape[1] * shape[2], int(seg[1])
    assert n == int(full[1]) - N and torch.equal(seg[0][:n], full[0][N:N + n])


def test_outputs_off_a_16_byte_boundary():
    X = to_device(corr_clip(6, 5, 7, 200, seed=9, dtype="bf16"))
    ref = P.ttf_compress(X, 1, 0.6, anchor_mode=1)
    L = int(ref[1])
    buf = torch.zeros(ref[0].numel() + 8, dtype=torch.bfloat16, device="cuda")
    tok = buf[1:1 + ref[0].numel()].view(ref[0].shape)
    _, cnt, pos = P.ttf_compress(X, 1, 0.6, out_tokens=tok, anchor_mode=1)
    assert int(cnt) == L and torch.equal(tok[:L], ref[0][:L]) and torch.equal(pos[:L], ref[2][:L])


@pytest.mark.parametrize("dtype", ["bf16", "f32"])
def test_a_wait_that_ran_out_is_reported_by_its_own_call(dtype):
    X = to_device(corr_clip(6, 5, 7, 256, seed=10, dtype=dtype))
    st = torch.cuda.Stream()
    ref = P.ttf_compress(X, 1, 0.6, anchor_mode=1, stream=st)
    L = int(ref[1])
    for _ in range(2):
        P.ttf_debug_set_wait(32, 16)
        try:
            _, cnt, _ = P.ttf_compress(X, 1, 0.6, anchor_mode=1, stream=st)
            assert P.ttf_last_device_status(st) == B.TTF_ERR_TIMEOUT and int(cnt) == -1
        finally:
            P.ttf_debug_set_wait()
        tok, cnt, pos = P.ttf_compress(X, 1, 0.6, anchor_mode=1, stream=st)
        assert P.ttf_last_device_status(st) == B.TTF_OK and int(cnt) == L
        assert torch.equal(tok[:L], ref[0][:L]) and torch.equal(pos[:L], ref[2][:L])
        tok, cnt, _ = P.ttf_compress(X, 1, 0.6, stream=st)
        assert P.ttf_last_device_status(st) == B.TTF_OK and int(cnt) > 0


def test_a_captured_call_replays():
    X = to_device(corr_clip(9, 8, 8, 256, seed=11, dtype="bf16"))
    ref = P.ttf_compress(X, 1, 0.6, anchor_mode=1)
    L = int(ref[1])
    st, outs = torch.cuda.Stream(), [torch.zeros_like(t) for t in ref]
    P.ttf_compress(X, 1, 0.6, *outs, anchor_mode=1, stream=st)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=st):
        for _ in range(3):
            P.ttf_compress(X, 1, 0.6, *outs, anchor_mode=1, stream=st)
    for _ in range(3):
        [t.zero_() for t in outs]
        g.replay()
        torch.cuda.synchronize()
        assert int(outs[1]) == L and torch.equal(outs[0][:L], ref[0][:L]) and torch.equal(outs[2][:L], ref[2][:L])
