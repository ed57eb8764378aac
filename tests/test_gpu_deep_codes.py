"""Recovery of streams whose rarest symbols have codes as long as the decode tables resolve, and one or two bits more,
placed where a lane's bit buffer is full: two such codes, then two of one bit, at a step that starts on a word of the
chunk. Whole chunks and the partial last one, one to four streams and a chain of six. Against the CPU oracle, bit for bit.
"""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

DEV = "cuda:0"
CHUNK, ROW, GROUP = 4096, 128, 4


@pytest.fixture(scope="module")
def lc():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2009_13003_b200 import binding

    binding.lib()
    return binding


def deep_deltas(depth, pairs, tail, seed):
    """Deltas of depth + 1 values, the counts of which give Huffman lengths 1, 2, ... depth, depth. In lane 0 of every
    chunk, which has one-bit codes otherwise, the two rarest stand side by side where the bits before them fill words."""
    rng = np.random.default_rng(seed)
    counts = pairs * np.array([1, 1] + [2 ** r for r in range(1, depth)], dtype=np.int64)
    values = np.ldexp(np.float32(1.0), -2 - np.arange(depth + 1)).astype(np.float32)
    n = int(counts.sum()) + tail  # a whole number of chunks, then a partial one
    counts[-1] += tail
    sym = np.full(n, -1, np.int64)
    sym[(np.arange(n) % ROW) < GROUP] = depth
    nchunks = (n + CHUNK - 1) // CHUNK
    for p, c in enumerate([nchunks - 1] + list(range(pairs - 1))):  # the partial chunk has one
        i = c * CHUNK + 8 * (p % 4) * ROW  # 4 bits a step: bit 0, 32, 64 or 96 of the chunk
        sym[i], sym[i + 1] = p % 2, 1 - p % 2
    left = counts - np.bincount(sym[sym >= 0], minlength=depth + 1)
    rest = np.repeat(np.arange(depth + 1), left)
    rng.shuffle(rest)
    sym[sym < 0] = rest
    return values[sym]


@pytest.mark.parametrize("depth,pairs", [(15, 40), (16, 24), (17, 12)])
def test_longest_table_codes_at_a_full_bit_buffer(lc, oracle, depth, pairs):
    streams, host = [], []
    for j in range(6):
        d = deep_deltas(depth, pairs, 3096, 70 + j)
        zero = np.zeros_like(d)
        lengths = sorted(int(x) for x in oracle.table(zero, d, 5)["len"] if x)
        assert lengths == list(range(1, depth + 1)) + [depth]
        host.append(oracle.compress(zero, d, 5))
        got = lc.compress(torch.from_numpy(zero).to(DEV), torch.from_numpy(d).to(DEV), 5)
        assert got.cpu().numpy().tobytes() == host[-1].tobytes()
        streams.append(got)
    base = np.random.default_rng(7).standard_normal(d.size).astype(np.float32)
    gbase = torch.from_numpy(base).to(DEV)
    for first, k in ((0, 1), (1, 1), (0, 2), (2, 3), (1, 4), (0, 6)):
        want = oracle.recover(base, host[first:first + k])
        got = lc.recover(gbase, streams[first:first + k]).cpu().numpy()
        bad = np.flatnonzero(got.view(np.uint32) != want.view(np.uint32))
        assert bad.size == 0, "%d streams from %d: %d elements differ, the first at %d" % (k, first, bad.size, bad[0])
