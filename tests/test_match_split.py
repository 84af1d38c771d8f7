"""How the tcgen05 matching kernel splits a launch: the parts of a tile's channel range depend on the clip alone, and are never
fewer than tiles of one grid row would have, whose sums in tensor memory the similarities' error stems from."""
import random

import pytest

import paper_2605_07355_b200 as P
from paper_2605_07355_b200 import build as B

SMS = 148


@pytest.fixture(scope="module", autouse=True)
def built():
    B.build()


def chunks_of_one_row_tiles(F, H, W, C, r):
    tiles, stages, n = -(-F // 32) * H * -(-W // 4), -(-C // 64), 1
    while n * 2 <= (4 if r == 2 else 8) and tiles * n * 2 <= 2 * SMS and stages // (n * 2) >= 2:
        n *= 2
    return n


def shapes(n):
    rng = random.Random(11)
    for _ in range(n):
        yield rng.choice([rng.randint(1, 9), rng.randint(1, 130)]), rng.randint(1, 33), rng.randint(1, 33), 8 * rng.randint(8, 512), rng.choice([0, 1, 1, 2])


def test_no_fewer_parts_than_in_tiles_of_one_row():
    seen = set()
    for s in list(shapes(4000)) + [(8, 8, 8, 4096, 1), (4, 12, 12, 4096, 1), (5, 12, 12, 2048, 1)]:
        rows, chunks, pieces = P.ttf_debug_match_split(*s)
        assert chunks >= chunks_of_one_row_tiles(*s), s
        seen.add((rows, chunks))
    assert {(w, c) for w in (1, 2, 4) for c in (1, 8)} <= seen


def test_the_parts_do_not_depend_on_the_launch():
    """... and a CTA keeps at most 256 columns of accumulators: two CTAs share the tensor memory of an SM"""
    for s in shapes(1000):
        one = P.ttf_debug_match_split(*s)
        for clips in (1, 2, 7, 16):
            rows, chunks, pieces = P.ttf_debug_match_split(*s, clips=clips, lanes=1 + clips % 2)
            assert chunks == one[1] and chunks % pieces == 0
            columns = -(-(4 + 2 * s[4]) * (rows + 2 * s[4]) // 16) * 16
            assert chunks // pieces * columns <= 256


def test_clips_of_other_kernels():
    assert P.ttf_debug_match_split(4, 8, 8, 56, 1) is None and P.ttf_debug_match_split(4, 8, 8, 64, 3) is None
    assert P.ttf_debug_match_split(4, 8, 8, 1001, 1) is None
    with pytest.raises(P.TTFError):
        P.ttf_debug_match_split(4, 8, 8, 64, 1, clips=17)
