"""What a plan's workspace holds beside its per-pair and per-entry arrays is
bounded by what the plan can use: digit counters for the blocks that its keys
fill, long lists only where it hands lists over."""

import math

import pytest


@pytest.fixture(scope="module")
def api():
    from paper_2602_23040_gb300 import api, build
    try:
        build.build()
    except RuntimeError as e:          # no nvcc on this machine
        pytest.skip(str(e))
    return api


def _beside_arrays(api, side, occ, sizes, **kw):
    """workspace_bytes less 44 bytes a pair, 12 an entry, the motion masks and the atlas's word offsets."""
    import synth
    views = [synth.scenes.pinhole((0, 0, -3), w, h) for w, h in sizes]
    p = api.Plan([(side, side, 0, 0, 0)], (side, side), 3, 1, "f32", views, int(occ * side * side), **kw)
    s = p.sizes
    words = s.mask_words * 33 // 32 + side * math.ceil(side / 32)
    return s.workspace_bytes - 44 * s.n_pairs - 12 * s.max_dups - 4 * words


RIG = [(1920, 1080), (1280, 720)] * 26
FIXED = 0.5e6       # block tables and sums, view tables, alignment
COUNTERS = 8 << 11  # of one block with 11-bit digits (8-bit ones: 256 of up to twice the blocks)
# a list handed over: per pixel of its 16 x 16 block 20 bytes forward and 8 backward, and 28 of its own; a segment: 8
# per pixel.  At most 4 x 152 lists, 64 segments of each of the first 128 and 16 of the others.
LIST, SEGMENT, MOST, MOST_SEGMENTS = 256 * 28 + 28, 256 * 8, 608, 128 * 64 + 480 * 16


@pytest.mark.parametrize("side,occ,sizes,blocks,hands", [
    (64, 1.0, [(256, 256)], 32 * 4096 // 2048, True),          # as many blocks as tiles of 2,048 entries
    (301, 0.57, [(641, 479)], 2 * 152, True),                  # one wave: two per SM
    (1024, 0.6, [(1920, 1080)], 2 * 152, True),
    (1024, 0.6, RIG, 4 * 2 * 152 + 52, False)])                # four waves, one more per view; 306 K work items
def test_workspace_beside_the_arrays(api, side, occ, sizes, blocks, hands):
    items = sum(math.ceil(w / 32) * math.ceil(h / 32) for w, h in sizes) * 4
    lists = min(items, MOST) * LIST + MOST_SEGMENTS * SEGMENT if hands else 0
    assert _beside_arrays(api, side, occ, sizes) <= blocks * COUNTERS + lists + FIXED


def test_segments_follow_the_entries(api):
    # 4 quadrants x 1,024 entries / 64 + 1 segments; one block's counters
    beside = _beside_arrays(api, 16, 0.1, [(640, 480)], max_dups=1024)
    assert beside <= COUNTERS + MOST * LIST + 65 * SEGMENT + FIXED


def test_counting_plan_shares_the_workspace(api):
    for sizes in ([(640, 480)], RIG):
        a, b = (_beside_arrays(api, 64, 1.0, sizes, count_evals=c) for c in (False, True))
        assert a == b
