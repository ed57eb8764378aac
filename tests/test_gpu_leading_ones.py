"""Recovery through the decoder's three forms of table: by 7 bits, by leading ones, and in two levels for codes which neither
index resolves. Codes of chosen lengths, mixed chains, chunks copied with and without space between the lanes, chunks larger
than the staging area, whole and partial ones; one to four streams and more. Against the CPU oracle, bit for bit.
"""
import numpy as np
import pytest
import torch

from test_gpu_parity import DEV, assert_recover_parity

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lc():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2009_13003_b200 import binding

    binding.lib()
    return binding


def deltas(weights, n, seed):
    """n values of len(weights) buckets, met in proportion to the weights."""
    rng = np.random.default_rng(seed)
    w = np.asarray(weights, np.float64)
    sym = rng.choice(w.size, size=n, p=w / w.sum())
    return (np.ldexp(1.0 + 0.5 * rng.random(n), -2 - sym // 2) * (1 - 2 * (sym % 2))).astype(np.float32)


SHAPES = {
    "two of one bit": ([1, 1], 2),  # 7 bits
    "four of two bits": ([1] * 4, 3),
    "sixteen of four bits": ([1] * 16, 5),
    "twenty of four and five bits": ([1] * 20, 5),
    "up to seven bits": ([1, 2, 4, 8, 12, 8, 4, 2, 1, 0.5, 0.1], 4),
    "up to eight bits": ([1, 2, 4, 8, 12, 8, 4, 2, 1, 0.5, 0.1, 0.1], 4),  # leading ones
    "two bits on average": ([8, 4, 2, 1, 0.5, 0.3, 0.2, 0.1, 0.05], 4),  # lanes near 8 words apart: copied with space
    "four bits on average": ([1, 2, 3, 4, 5, 6, 7, 8, 8, 7, 6, 5, 4, 3, 2, 1, 0.5, 0.2, 0.1, 0.02], 5),  # near 16 words
    "long tail": ([2.0 ** -i for i in range(15)], 4),  # up to 14 bits
    "two hundred of seven and eight bits": ([1] * 200, 8),  # two levels
}


def test_the_shapes_are_what_they_say(oracle):
    def bits(name):
        w, nbits = SHAPES[name]
        d = deltas(w, 1 << 18, 3)
        t = oracle.table(np.zeros_like(d), d, nbits)
        ln = np.asarray(t["len"], np.int64)
        sym = oracle.symbols(np.zeros_like(d), d, nbits)
        return sorted(set(ln[np.unique(sym)])), ln[sym].mean()

    for name, lengths in (("four of two bits", [2]), ("sixteen of four bits", [4]), ("twenty of four and five bits", [4, 5]),
                          ("up to seven bits", list(range(2, 8))), ("up to eight bits", list(range(2, 9))), ("long tail", list(range(1, 15))),
                          ("two hundred of seven and eight bits", [7, 8])):
        assert bits(name)[0] == lengths, name
    # the copy leaves space where 128 codes are within 0.6 words of a multiple of 8 words; a chunk's bytes are rounded up to 16
    for name, spaced in (("two bits on average", True), ("four bits on average", True), ("up to eight bits", False)):
        words = bits(name)[1] * 128 / 32
        assert (abs(words / 8 - round(words / 8)) * 8 < 0.5) == spaced, (name, words)


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("n", [3, 4096, 5 * 4096 + 1, 40 * 4096 + 2777])
def test_code_shapes(lc, oracle, shape, n):
    weights, nbits = SHAPES[shape]
    base = torch.from_numpy(np.random.default_rng(9).standard_normal(n).astype(np.float32)).to(DEV)
    streams = [oracle.compress(np.zeros(n, np.float32), deltas(weights, n, 20 + j), nbits) for j in range(4)]
    for k in (1, 2, 3, 4):
        assert_recover_parity(lc, oracle, base, streams[:k], inplace=k % 2 == 0)


def test_mixed_chains(lc, oracle):
    n = 9 * 4096 + 130
    zero = np.zeros(n, np.float32)
    base = torch.from_numpy(np.random.default_rng(9).standard_normal(n).astype(np.float32)).to(DEV)
    streams = [oracle.compress(zero, deltas(SHAPES[s][0], n, 30 + j), SHAPES[s][1]) for j, s in enumerate(SHAPES)]
    fixed = oracle.compress(zero, deltas([1] * 30, n, 40), 8, fixed=True)
    for chain in (streams[:4], streams[4:8], streams[5:7] + streams[2:3], [fixed, streams[1]], [fixed, streams[8]], streams[3:] + [fixed],
                  [fixed] * 3, streams[:3] + [fixed], streams[9:] + streams[:3], [streams[9]] * 4):
        assert_recover_parity(lc, oracle, base, chain)


@pytest.mark.parametrize("k", [1, 2, 3, 4])
@pytest.mark.parametrize("shape", ["four bits on average", "long tail", "up to seven bits", "two hundred of seven and eight bits"])
def test_chunks_larger_than_the_staging_area(lc, oracle, shape, k):
    # the rarest bucket fills chunks of its own: some are several times the average
    weights, nbits = SHAPES[shape]
    n = 300 * 4096 + 1000
    d = deltas(weights, n, 50)
    rare = d[np.argmin(np.abs(d))]
    for c in (0, 7, 299):
        d[c * 4096:(c + 1) * 4096] = rare
    d[-1000:] = rare
    base = torch.from_numpy(np.random.default_rng(9).standard_normal(n).astype(np.float32)).to(DEV)
    stream = oracle.compress(np.zeros(n, np.float32), d, nbits)
    assert_recover_parity(lc, oracle, base, [stream] * k)
