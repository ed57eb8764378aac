"""How the per-layer recovery deals its segments out to CTAs (host code, no GPU): every segment has its share, also when
there are about as many segments as the device holds CTAs.
"""
import ctypes as C
import random

import pytest

CHUNK = 4096


def split(sizes, warps, slots):
    from paper_2009_13003_b200 import binding

    begin = [0]
    for s in sizes:
        begin.append(begin[-1] + s)
    out = (C.c_uint32 * (len(sizes) + 1))()
    ctas = binding.lib().lc_debug_split_segments((C.c_uint64 * len(begin))(*begin), len(sizes), warps, slots, out)
    assert out[0] == 0 and out[len(sizes)] == ctas > 0
    return [b - a for a, b in zip(out[:-1], out[1:])]


def rounds(size, warps):
    return max(1, -(-(-(-size // CHUNK)) // warps))


def makespan(sizes, shares, warps, slots):
    """In rounds, preparation (half a round) included, the CTAs started in order as slots come free."""
    import heapq

    free = [0.0] * slots
    for size, ctas in zip(sizes, shares):
        for _ in range(ctas):
            heapq.heapreplace(free, free[0] + 0.5 + -(-rounds(size, warps) // ctas))
    return max(free)


# (warps, slots) of launches with one, two and four streams on 148 SMs
SHAPES = [(12, 296), (20, 148), (16, 148)]
SKEWED = {
    "130, of which 30 of 600 chunks": [600 * CHUNK] * 30 + [1000] * 100,
    "148 and a large one": [4000] * 148 + [25_000_000],
    "149 and a large one first": [25_000_000] + [4000] * 149,
    "159 and a large one": [4000] * 159 + [300_000_000],
    "160 of two sizes": [4096, 2_000_000] * 80,
    "140 and a large one": [64] * 140 + [40_000_000],
}


@pytest.mark.parametrize("warps,slots", SHAPES)
@pytest.mark.parametrize("name", SKEWED)
def test_large_segments_have_their_share(name, warps, slots):
    sizes = SKEWED[name]
    shares = split(sizes, warps, slots)
    work = sum(0.5 + rounds(s, warps) for s in sizes) / slots
    # twice the work spread evenly, and the preparations and partial rounds of a few waves
    assert makespan(sizes, shares, warps, slots) <= 2.0 * work + 4.0, (max(shares), work)


@pytest.mark.parametrize("warps,slots", SHAPES)
def test_one_wave_stays_one_wave(warps, slots):
    from paper_2009_13003_b200 import synth

    # a model that fits in one wave of single rounds, or of a few: the smallest number of rounds that fits
    for sizes in ([100_000] * 20, synth.resnet18_segments(), [4096] * 140, [0, 4, 8, 0]):
        shares = split(sizes, warps, slots)
        assert sum(shares) <= slots
        r = max(-(-rounds(s, warps) // c) for s, c in zip(sizes, shares))
        if r > 1:
            assert sum(-(-rounds(s, warps) // (r - 1)) for s in sizes) > slots


def test_every_chunk_has_a_warp_and_no_cta_is_idle():
    rng = random.Random(5)
    for _ in range(200):
        sizes = [4 * rng.choice([0, 1, 1000, 1024, 1025, rng.randint(1, 1 << rng.randint(1, 24))]) for _ in range(rng.randint(1, 160))]
        for warps, slots in SHAPES:
            for s, c in zip(sizes, split(sizes, warps, slots)):
                assert 1 <= c <= rounds(s, warps)
