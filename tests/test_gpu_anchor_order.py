"""The anchor does not depend on the launch: clips whose frames hold the same tokens in another order have mean tokens that are
equal but for the order of summation, so the arg max falls where the last bits say.  Alone, in a batch of any size and under
every schedule the same frame has to win."""
import pytest
import torch

import paper_2605_07355_b200 as P

pytestmark = pytest.mark.gpu


def shuffled_frames(F, H, W, C, dtype, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    base = torch.randn((H * W, C), generator=g, device="cuda")
    base *= torch.exp(2 * torch.randn((H * W, 1), generator=g, device="cuda"))       # (norms over decades: sums that round)
    frames = [base[torch.randperm(H * W, generator=g, device="cuda")] for _ in range(F)]
    return torch.stack(frames).view(F, H, W, C).to(dtype)


def anchors_of_batch(Xs):
    _, _, pos = P.ttf_compress_batch(Xs, 1, 0.6)
    torch.cuda.synchronize()
    return [int(p[0, 0]) for p in pos]                       # the first row is a token of the anchor frame


# slices of 8 lanes alone and 16 or 32 in a batch, of 16 alone and 32 in a batch; statistics over one to 32 slices (eight or
# sixteen CTAs), more frames than one chunk; both data types
@pytest.mark.parametrize("shape,dtype", [((8, 16, 16, 1024), "bf16"), ((32, 9, 9, 1024), "bf16"), ((16, 12, 12, 2048), "bf16"),
                                         ((32, 6, 6, 4096), "bf16"), ((70, 15, 15, 1160), "bf16"), ((6, 20, 21, 72), "bf16"),
                                         ((12, 11, 13, 640), "f32"), ((40, 6, 6, 1152), "f32")])
def test_near_ties_fall_the_same_way_alone_and_in_batches(shape, dtype):
    dt = torch.float32 if dtype == "f32" else torch.bfloat16
    Xs = [shuffled_frames(*shape, dt, seed) for seed in range(48)]
    alone = [int(P.ttf_query(X, 1, 0.6, want=("anchor",))["anchor"]) for X in Xs]
    assert len(set(alone)) > 1                               # (the last bits do decide)
    for n in (2, 6, 16, 48):
        got = [a for i in range(0, 48, n) for a in anchors_of_batch(Xs[i:i + n])]
        assert got == alone, n
    try:
        for schedule in (1, 3, 8, P.TTF_SCHEDULE_PIPELINED):
            P.ttf_set_schedule(schedule)
            assert anchors_of_batch(Xs[:16]) == alone[:16], schedule
    finally:
        P.ttf_set_schedule(0)


@pytest.mark.parametrize("C,slices", [(256, (0, 1)), (384, (0, 2)), (512, (0, 1)), (512, (1, 2)), (640, (0, 4))])
def test_small_shares_of_one_slice_are_not_lost_in_a_large_one_of_another(C, slices):
    """One token per frame.  Frame 1 is frame 0 (its square is beyond 2^23, where a step of fp32 in the product with the sum of all
    frames is 2) and four small channels in another slice of 128, whose four shares of 0.9 each would not count one by one.  They make
    its cosine the larger one by 2e-7; everything else is exact."""
    large, small = slices
    X = torch.zeros((3, 1, 1, C), dtype=torch.float32)
    X[0, 0, 0, large * 128] = X[1, 0, 0, large * 128] = 2900.0
    few = slice(small * 128, small * 128 + 4)
    X[1, 0, 0, few] = 0.9 / 64
    X[2, 0, 0, few] = 64.0
    assert int(P.ttf_query(X.cuda(), 0, 0.6, want=("anchor",))["anchor"]) == 1
