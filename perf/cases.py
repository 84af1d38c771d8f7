"""The work a user of the library has it do, as cases that can be timed.

A video-language program holds the visual tokens of a clip on the GPU (the projector's output) and calls the pass
before prefill; a server does so for the clips of several requests at once; a streaming program compresses the new
frames of a segment against the last frame it kept; a program that calibrates its threshold looks at the decisions
without the gather; a decoder that needs the full grid restores it; a program whose tokens live in host memory uses
the host entry point.  Sizes are those of the synthetic workloads in paper_2605_07355_b200/clips.py, of the tests,
and ragged ones between them.

Inputs follow the anchored generator of clips.py (one base scene, a small cumulative camera shift per frame,
LogNormal token scale), made on the GPU.  A token is either static (cosine with the base scene 0.93 to 0.995) or
changed (0 to 0.5), and the share of changed tokens differs from frame to frame, so that about two thirds of the
tokens are fused at t = 0.70.  No similarity comes near t and no two frames tie for the anchor: another order of
summation takes the same decisions, and every output row is a bit copy of an input row.
"""
import math

import torch

import paper_2605_07355_b200 as P
from paper_2605_07355_b200 import accounting

CALM, BUSY = 0.05, 0.50          # share of changed tokens in the calmest and in the busiest frame


def _case(kind, F, H, W, C, dtype="bf16", r=1, t=0.70, clips=1, anchor=0, order=0, pos_base=0):
    return {"kind": kind, "F": F, "H": H, "W": W, "C": C, "dtype": dtype, "r": r, "t": t, "clips": clips,
            "anchor": anchor, "order": order, "pos_base": pos_base}


def listed():
    return [
        # a handful of frames on a small grid, fp32: the cost of a call as such
        dict(_case("compress", 4, 8, 8, 64, "f32"), name="tiny_f32"),
        # frames, grid and channels that fit no tile; the first frame as anchor, rows in natural order at an offset
        # (how a program that splices visual tokens into a prompt calls it)
        dict(_case("compress", 21, 13, 19, 1160, anchor=1, order=1, pos_base=35), name="ragged_options"),
        # one clip for a 2B-class model
        dict(_case("compress", 32, 16, 16, 2048), name="clip_c2048"),
        # one clip for an 8B-class model: the shape bench.py reports
        dict(_case("compress", 32, 16, 16, 4096), name="clip_c4096"),
        # a serving batch of such clips in one call: what bench.py times
        dict(_case("batch", 32, 16, 16, 4096, clips=16), name="batch_c4096"),
        # the long-video batch
        dict(_case("batch", 128, 16, 16, 4096, clips=8), name="batch_long"),
        # a high-resolution clip with the 5 x 5 window
        dict(_case("compress", 64, 32, 32, 4096, r=2), name="clip_wide_r2"),
        # a clip whose tokens were kept in fp32, at the width of a vision encoder
        dict(_case("compress", 32, 16, 16, 1152, "f32"), name="clip_f32"),
        # streaming: the rolling anchor and eight new frames; the caller needs the count before it can go on
        dict(_case("segment", 9, 16, 16, 4096, anchor=1), name="segment_c4096"),
        # the decisions without the gather, and their counts: choosing a threshold
        dict(_case("query", 48, 14, 14, 2048), name="query_c2048"),
        # back to the full grid, for a consumer that needs every position
        dict(_case("restore", 32, 16, 16, 4096), name="restore_c4096"),
        # tokens in pinned host memory, four clips through the pipelined host path
        dict(_case("host", 32, 16, 16, 4096, clips=4), name="host_c4096"),
    ]


MOST_BYTES = 512 << 20           # input bytes of a drawn device case (the long-video batch has four times as many)
MOST_HOST_BYTES = 128 << 20


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["compress"] * 5 + ["batch"] * 3 + ["segment"] * 2 + ["query", "restore", "host"])
    dtype = "f32" if kind in ("compress", "batch", "query") and rng.random() < 0.2 else "bf16"
    H, W = log_int(6, 32), log_int(6, 32)
    C = 8 * log_int(8, 512)                                     # 64 .. 4096 channels
    F = log_int(3, 24) if kind == "segment" else log_int(4, 128)
    clips = log_int(2, 16) if kind == "batch" else (log_int(1, 6) if kind == "host" else 1)
    r = rng.choice([0, 1, 1, 1, 1, 2])
    t = rng.choice([0.65, 0.70, 0.70, 0.80])
    anchor = 1 if kind == "segment" or (kind in ("compress", "batch") and rng.random() < 0.2) else 0
    order = 1 if anchor and kind != "segment" and rng.random() < 0.5 else 0
    most = MOST_HOST_BYTES if kind == "host" else MOST_BYTES // (4 if dtype == "f32" else 1)
    size = lambda: F * H * W * C * (4 if dtype == "f32" else 2) * clips
    while size() > most:                                        # too large: fewer clips, then fewer frames
        if clips > 2:
            clips //= 2
        elif F > 8:
            F = F * 2 // 3
        else:
            C = max(64, C // 16 * 8)
    return _case(kind, F, H, W, C, dtype, r, t, clips, anchor, order, rng.randrange(100) if order else 0)


def _clip(case, seed):
    """One clip [F, H, W, C] on the GPU."""
    F, H, W, C = case["F"], case["H"], case["W"], case["C"]
    dev = torch.device("cuda")
    g = torch.Generator(device=dev)
    g.manual_seed(seed)
    host = torch.Generator()
    host.manual_seed(seed)
    shift = max(1, min(2, case["r"]))
    steps = torch.randint(-shift, shift + 1, (F, 2), generator=host).tolist()
    busy = torch.linspace(CALM, BUSY, F)[torch.randperm(F, generator=host)].tolist()
    out = torch.empty((F, H, W, C), dtype=torch.float32 if case["dtype"] == "f32" else torch.bfloat16, device=dev)
    base = torch.randn((H, W, C), generator=g, device=dev)
    moved = torch.rand((F, H, W, 1), generator=g, device=dev)
    how_far = torch.rand((F, H, W, 1), generator=g, device=dev)
    scale = torch.exp(0.2 * torch.randn((F, H, W, 1), generator=g, device=dev))
    oy = ox = 0
    for k in range(F):
        if k > 0:                                               # cumulative shift inside [0, shift]^2
            oy, ox = min(max(oy + steps[k][0], 0), shift), min(max(ox + steps[k][1], 0), shift)
        cos = torch.where(moved[k] < busy[k], 0.5 * how_far[k], 0.93 + 0.065 * how_far[k])
        noise = torch.randn((H, W, C), generator=g, device=dev)
        x = torch.roll(base, (oy, ox), (0, 1)) * (cos * scale[k]) + noise * (torch.sqrt(1 - cos * cos) * scale[k])
        out[k].copy_(x)
    return out


def _buffers(case, n):
    """The output buffers a program keeps: room for every token, one set per clip."""
    rows, C = case["F"] * case["H"] * case["W"], case["C"]
    dt = torch.float32 if case["dtype"] == "f32" else torch.bfloat16
    return ([torch.zeros((rows, C), dtype=dt, device="cuda") for _ in range(n)],
            [torch.zeros(1, dtype=torch.int32, device="cuda") for _ in range(n)],
            [torch.zeros((rows, 3), dtype=torch.int32, device="cuda") for _ in range(n)])


def prepare(case, seed):
    kind, n = case["kind"], case["clips"]
    clips = [_clip(case, seed * 64 + j) for j in range(n)]
    s = {"case": case}
    if kind in ("compress", "batch"):
        s["clips"], s["out"] = clips, _buffers(case, n)
    elif kind == "segment":
        s["clips"] = clips
        s["cache"], _, s["cache_pos"] = (b[0] for b in _buffers(case, 1))
    elif kind == "query":
        s["clips"] = clips
    elif kind == "restore":
        q = P.ttf_query(clips[0], case["r"], case["t"], want=("anchor", "keep", "dst"))
        tok, cnt, _ = P.ttf_compress(clips[0], case["r"], case["t"])
        s["tokens"], s["query"] = tok[:int(cnt)].clone(), q
    elif kind == "host":
        rows = case["F"] * case["H"] * case["W"]
        s["clips"] = [c.cpu().pin_memory() for c in clips]
        s["tok"] = [torch.zeros((rows, case["C"]), dtype=c.dtype).pin_memory() for c in clips]
        s["pos"] = [torch.zeros((rows, 3), dtype=torch.int32).pin_memory() for c in clips]
    return s


def run(s):
    case = s["case"]
    kind, r, t = case["kind"], case["r"], case["t"]
    if kind == "compress":
        tok, cnt, pos = s["out"]
        return P.ttf_compress(s["clips"][0], r, t, tok[0], cnt[0], pos[0], anchor_mode=case["anchor"],
                              order=case["order"], pos_base=case["pos_base"])
    if kind == "batch":
        return P.ttf_compress_batch(s["clips"], r, t, *s["out"], anchor_mode=case["anchor"], order=case["order"],
                                    pos_base=case["pos_base"])
    if kind == "segment":
        tok, cnt, pos = P.ttf_compress_segment(s["clips"][0], r, t, frame_base=16)
        n = int(cnt)                                            # this many new tokens join the stream so far
        s["cache"][:n] = tok[:n]
        s["cache_pos"][:n] = pos[:n]
        return s["cache"], n, s["cache_pos"]
    if kind == "query":
        q = P.ttf_query(s["clips"][0], r, t)
        q["stats"] = P.ttf_stats(q["best_sim"], q["keep"], q["anchor"], case["F"], case["H"], case["W"], t)
        return q
    if kind == "restore":
        q = s["query"]
        return P.ttf_restore(s["tokens"], case["F"], case["H"], case["W"], q["anchor"], q["keep"], q["dst"])
    _, counts, _ = P.ttf_compress_host_batch(s["clips"], r, t, s["tok"], s["pos"])
    return s["tok"], counts, s["pos"]


def work(case):
    """Input read once, output written once, and the multiply-adds of the window search.  The number of kept tokens is
    the generator's expectation: a source token is fused when neither it nor its anchor cell has changed."""
    F, H, W, C, n = case["F"], case["H"], case["W"], case["C"], case["clips"]
    N, item = H * W, 4 if case["dtype"] == "f32" else 2
    row = C * item
    anchor_changed = CALM if case["anchor"] == 0 else (CALM + BUSY) / 2
    kept = (F - 1) * N * (1 - (1 - (CALM + BUSY) / 2) * (1 - anchor_changed))
    kept += 0 if case["kind"] == "segment" else N
    if case["kind"] == "restore":
        return {"bytes": kept * row + F * N * (row + 4 + 4 + 1), "flops": 0}
    if case["kind"] == "query":
        out = F * N * (1 + 4 + 4) + N * 4
    else:
        out = kept * (row + 12) + 4
    return {"bytes": n * (F * N * row + out), "flops": n * accounting.matching_flops(F, H, W, C, case["r"])}


def tolerance(case):
    if case["kind"] == "query":
        # the similarities are sums of C products in fp32, in an order of the kernel's choice; a destination may
        # differ where a changed token is equally unlike two cells of its window
        return {"rel": 1e-5, "max": 1e-4, "differ": 5e-4}
    return "exact"                                              # bit copies, positions and counts
