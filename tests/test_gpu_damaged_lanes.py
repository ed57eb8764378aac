"""Recovery from streams whose lane index and payload are damaged, through every way a chunk can take: the three forms of table, the copy
with and without space, chunks larger than the staging area. What comes out is unspecified, but the status is one of two, nothing
beside the output is written, and the next call is unharmed. (No read leaves its chunk: lane starts are clamped to it, in shared memory a
lane moves at most 1013 bytes on, within the launch's padding, and words read from global memory end with the chunk.)
"""
import numpy as np
import pytest
import torch

from test_gpu_leading_ones import SHAPES, deltas
from test_gpu_parity import DEV, assert_recover_parity

pytestmark = pytest.mark.gpu

# "long tail" with chunks of its rarest bucket: larger than the staging area
CASES = ["twenty of four and five bits", "up to seven bits", "two bits on average", "up to eight bits", "long tail",
         "two hundred of seven and eight bits"]


def damaged(stream, how, rng):
    """The stream with every third chunk's lane bit counts, and some payload, replaced; header, table and chunk index stay valid."""
    m = stream.copy()
    nsym, nchunks = (int(np.frombuffer(m[o:o + 4].tobytes(), "<u4")[0]) for o in (16, 32))
    lanes = 64 + 16 * nsym + 8 * (nchunks + 1)
    payload = int(np.frombuffer(m[56:64].tobytes(), "<u8")[0])
    for c in range(0, nchunks, 3):
        row = m[lanes + 64 * c: lanes + 64 * (c + 1)]
        row[:] = {"saturated": 0xFF, "zero": 0, "random": rng.integers(0, 256, 64, dtype=np.uint8)}[how]
    span = m[payload + (m.size - payload) // 3: payload + (m.size - payload) // 2]
    span[:] = 0xFF if how == "saturated" else rng.integers(0, 256, span.size, dtype=np.uint8)
    return m


@pytest.mark.parametrize("how", ["saturated", "zero", "random"])
@pytest.mark.parametrize("shape", CASES)
def test_damaged_lane_index(oracle, shape, how):
    from paper_2009_13003_b200 import binding as lc

    rng = np.random.default_rng(17)
    weights, nbits = SHAPES[shape]
    n, pad = 60 * 4096 + 1000, 1024
    d = deltas(weights, n, 60)
    if shape == "long tail":
        rare = d[np.argmin(np.abs(d))]
        for c in (0, 3, 59):
            d[c * 4096:(c + 1) * 4096] = rare
    good = oracle.compress(np.zeros(n, np.float32), d, nbits)
    bad = torch.from_numpy(damaged(good, how, rng)).to(DEV)
    good_t = torch.from_numpy(good).to(DEV)
    base = torch.from_numpy(rng.standard_normal(n).astype(np.float32)).to(DEV)
    ws = lc.alloc_workspace(0, DEV)
    for k in (1, 2, 3, 4):
        out = torch.full((n + pad,), 7.0, device=DEV)
        streams = [good_t] * (k - 1) + [bad]
        lc.recover_async(base, streams, out[:n], ws)
        assert lc.last_status(ws) in (lc.OK, lc.ERR_FORMAT)
        assert bool((out[n:] == 7.0).all()), "written beyond the output"
        assert torch.equal(good_t.cpu(), torch.from_numpy(good))
        assert_recover_parity(lc, oracle, base, [good] * k)
