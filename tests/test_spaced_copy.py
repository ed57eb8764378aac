"""The units that the decoder copies of a chunk with space between the lanes, restated in numpy: whatever the lane index says, every
unit read lies in the chunk, every unit written in its area, no unit is written twice, and each group of four lanes finds the units
that its codes lie in. CPU only; the kernel itself meets damaged lane indices in test_gpu_damaged_lanes.py.
"""
import numpy as np
import pytest

UNIT, GROUPS = 16, 8


def copied(lane_bits, nbytes):
    """[(group, source unit, destination unit)] and the lanes' starts, in bits, as the kernel computes them."""
    start = np.minimum(np.cumsum(lane_bits) - lane_bits, nbytes * 8)
    units = nbytes // UNIT
    out = []
    for g in range(GROUPS):
        first = start[4 * g] >> 7
        end = units if g == GROUPS - 1 else min((start[4 * g + 4] >> 7) + 1, units)
        out += [(g, u, u + g) for u in range(first, end)]
    return out, start


@pytest.mark.parametrize("kind", ["valid", "random", "saturated", "zero", "large first"])
def test_every_unit_stays_inside(kind):
    rng = np.random.default_rng(3)
    for _ in range(200):
        valid = rng.integers(100, 160, 32)
        nbytes = int(-(-int(valid.sum()) // 128) * 16)
        bits = {"valid": valid, "random": rng.integers(0, 65536, 32), "saturated": np.full(32, 65535), "zero": np.zeros(32, np.int64),
                "large first": np.concatenate([[65535], valid[1:]])}[kind]
        moves, start = copied(bits, nbytes)
        assert all(0 <= u < nbytes // UNIT and u <= to < (nbytes + 7 * UNIT) // UNIT for _, u, to in moves)
        assert len({to for _, _, to in moves}) == len(moves)
        if kind == "valid":
            have = {(g, u) for g, u, _ in moves}
            for lane in range(32):
                end = start[lane] + bits[lane] - 1
                assert all((lane // 4, u) in have for u in range(start[lane] >> 7, (end >> 7) + 1))
