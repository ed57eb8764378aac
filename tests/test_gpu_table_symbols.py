"""The table pass compares symbols 32 at a time: numbers of used symbols around multiples of 32 and of the 16 warps, with equal counts, rising
ones and codes beyond 31 bits, for one vector and for a shard of one (whose weights are 64 bits), against the CPU oracle. Bar: byte-identical streams."""
import numpy as np
import pytest
import torch

from test_gpu_parity import DEV, to_np

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lc():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2009_13003_b200 import binding

    binding.lib()
    return binding


def _fib(count):
    a = [1, 1]
    while len(a) < count:
        a.append(a[-1] + a[-2])
    return a[:count]


@pytest.mark.parametrize("symbols,counts", [(s, c) for s in (2, 15, 16, 17, 31, 32, 33, 63, 65, 200) for c in ("equal", "rising")] +
                         [(s, "fibonacci") for s in (24, 33, 35)])
def test_codes_of(lc, oracle, symbols, counts):
    # exponent fields 20 .. 119, both signs; `symbols` buckets
    keys = [(e, s) for e in range(119, 19, -1) for s in (0, 1)][:symbols]
    weight = {"equal": [700] * symbols, "rising": [3 * (i // 2) + 1 for i in range(symbols)], "fibonacci": _fib(symbols) if counts == "fibonacci" else None}[counts]
    mantissa = 0x12345
    bits = np.concatenate([np.full(w, (s << 31) | (e << 23) | mantissa, np.uint32) for (e, s), w in zip(keys, weight)])
    delta = bits.view(np.float32)[np.random.default_rng(symbols).permutation(len(bits))] if len(bits) < 1 << 22 else bits.view(np.float32)
    cur = torch.from_numpy(delta.copy()).to(DEV)
    base = torch.zeros_like(cur)
    nbits = 8 if symbols < 200 else 9
    want = oracle.compress(to_np(base), to_np(cur), nbits)
    assert lc.compress(base, cur, nbits).cpu().numpy().tobytes() == want.tobytes()
    if len(bits) > 32 * 4096:
        ws = lc.alloc_workspace(cur.numel(), DEV)
        shard = lc.shard_encode(base, cur, nbits, lc.shard_stats(base, cur, ws), ws).cpu().numpy()
        same = want.copy()
        same[7] |= 2  # the flag of a shard; a vector that is its only shard has the same counts
        assert shard.tobytes() == same.tobytes()
