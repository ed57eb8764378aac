"""Recovery of chunks copied with space between the lanes and without, and of vectors that have both: the lanes' distance lies near a
multiple of 8 words. Against the CPU oracle, bit for bit.
"""
import numpy as np
import pytest
import torch

from test_gpu_leading_ones import deltas
from test_gpu_parity import DEV, assert_recover_parity

pytestmark = pytest.mark.gpu

# weights, nbits, a chunk's bytes less the nearest multiple of 1024
SHAPES = [([1] * 15, 5, -34), ([1] * 15 + [0.5], 5, 0), ([1] * 16 + [0.02], 5, 40), ([1] * 16 + [0.3], 5, 48), ([1] * 60, 8, -31)]


@pytest.mark.parametrize("weights,nbits,off", SHAPES)
def test_chunks_near_a_multiple_of_eight_words_a_lane(oracle, weights, nbits, off):
    from paper_2009_13003_b200 import binding as lc

    n = 40 * 4096 + 1234
    base = torch.from_numpy(np.random.default_rng(9).standard_normal(n).astype(np.float32)).to(DEV)
    streams = [oracle.compress(np.zeros(n, np.float32), deltas(weights, n, 120 + j), nbits) for j in range(4)]
    nsym = int(np.frombuffer(streams[0][16:20].tobytes(), "<u4")[0])
    index = np.frombuffer(streams[0][64 + 16 * nsym : 64 + 16 * nsym + 8 * 41].tobytes(), "<u8").astype(np.int64)
    near = (np.diff(index) + 512) % 1024 - 512
    assert abs(near.mean() - off) < 16
    for k in (1, 2, 3, 4):
        assert_recover_parity(lc, oracle, base, streams[:k], inplace=k % 2 == 1)
