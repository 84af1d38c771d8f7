"""ttf_restore and ttf_stats take no [F, H, W, C] clip whose device the binding checks, so they check their operands
themselves: host tensors are a ValueError before anything is allocated or launched, a missing one the library's error."""
import pytest
import torch

import paper_2605_07355_b200 as P


def operands(device):
    """F = 2, H = 1, W = 3; the anchor is frame 0, one token of frame 1 is kept"""
    return dict(compressed=torch.arange(8, dtype=torch.float32, device=device).view(4, 2),
                sim=torch.tensor([1, 1, 1, 0.9, 0.2, 0.8], dtype=torch.float32, device=device),
                anchor=torch.zeros(1, dtype=torch.int32, device=device),
                keep=torch.tensor([1, 1, 1, 0, 1, 0], dtype=torch.uint8, device=device),
                dst=torch.tensor([0, 1, 2, 0, 1, 2], dtype=torch.int32, device=device))


def restore(o):
    return P.ttf_restore(o["compressed"], 2, 1, 3, o["anchor"], o["keep"], o["dst"])


def stats(o):
    return P.ttf_stats(o["sim"], o["keep"], o["anchor"], 2, 1, 3, 0.5)


def test_host_tensors_are_refused():
    o = operands("cpu")
    with pytest.raises(ValueError):
        restore(o)
    with pytest.raises(ValueError):
        stats(o)


@pytest.mark.gpu
@pytest.mark.parametrize("name", ["anchor", "keep", "dst"])
def test_one_host_tensor_or_none_is_refused(name):
    calls = [restore] if name == "dst" else [restore, stats]
    for call in calls:
        o = operands("cuda")
        o[name] = o[name].cpu()
        with pytest.raises(ValueError):
            call(o)
        o[name] = None
        with pytest.raises(P.TTFError):
            call(o)


@pytest.mark.gpu
def test_pinned_host_arrays_are_still_taken():
    o = operands("cuda")
    for name in ("anchor", "keep", "dst"):
        o[name] = o[name].cpu().pin_memory()
    full, idx = restore(o)
    assert idx.tolist() == [0, 1, 2, 0, 3, 2]
    assert torch.equal(full.cpu(), o["compressed"].cpu()[[0, 1, 2, 0, 3, 2]])
    assert stats(o).tolist() == [1, 2, 0]
