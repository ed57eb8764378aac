"""How many warps of an SM the recovery of a flat vector gets (host code, no GPU): as many as hold its average chunks with some
room. The bytes of space that some chunks are copied with must not cost warps: where they are asked for, they fit beside.
"""
import pytest

ROOM = 227 * 1024 - 1024 - 1024 - 128  # shared memory without what the system and the launch set aside
TABLES = 2 * 8192 + 4000               # a stream's tables and state
MOST = {1: 24, 2: 20, 3: 20, 4: 16}    # by registers
REGS = {1: 80, 2: 96, 3: 96, 4: 128}


@pytest.mark.parametrize("k", [1, 2, 3, 4])
def test_as_many_warps_as_hold_average_chunks(k):
    from paper_2009_13003_b200 import binding

    for chunk in range(256, 4600, 8):
        area = -(-(chunk + chunk // 32 + 48) // 16) * 16
        fit = (ROOM - k * TABLES) // (k * area) if k > 1 else MOST[k]  # one stream: two CTAs of 12, with room to spare
        want = max(8, min(MOST[k], fit // 4 * 4))
        assert binding.lib().lc_debug_decode_warps(k, chunk, REGS[k]) == want, chunk


def test_bad_arguments():
    from paper_2009_13003_b200 import binding

    for k, regs in ((0, 96), (5, 96), (2, 0), (2, 256)):
        assert binding.lib().lc_debug_decode_warps(k, 2000, regs) == 0
