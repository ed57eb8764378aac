"""Vectors with a few deltas of 2 and more, which the one-byte key plane does not identify: only the chunks that hold one form their keys from base
and cur. Streams and tracked states against the CPU oracle, with such elements at the edges of chunks, in the partial last chunk, beside unchanged elements
(delta +0) and negative zeros, through every scan and with the state advanced in place."""
import numpy as np
import pytest
import torch

from test_gpu_parity import DEV, to_np
from test_gpu_update import check_update

pytestmark = pytest.mark.gpu
N = 41 * 4096 + 1234


@pytest.fixture(scope="module")
def lc():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2009_13003_b200 import binding

    binding.lib()
    return binding


CASES = {
    "first": ([0], 3.0), "last": ([N - 1], -2.0), "edges": ([4095, 4096, 40 * 4096 - 1, 41 * 4096 - 1], 1e6),
    "partial": ([41 * 4096, N - 2], -7.5), "one chunk": (list(range(8192, 12288)), 2.5), "every chunk": (list(range(100, N, 4096)), -1e30),
}


@pytest.mark.parametrize("nbits", [2, 5, 9])
@pytest.mark.parametrize("where", list(CASES))
def test_few_large_deltas(lc, oracle, where, nbits):
    rng = np.random.default_rng(nbits)
    base = rng.normal(0, 0.02, N).astype(np.float32)
    cur = base + (rng.normal(0, 1e-3, N) * np.exp2(-rng.integers(0, 12, N))).astype(np.float32)
    cur[5 * 4096:9 * 4096 + 7] = base[5 * 4096:9 * 4096 + 7]  # unchanged
    base[20 * 4096:20 * 4096 + 500], cur[20 * 4096:20 * 4096 + 500] = 0.0, -0.0  # a delta of -0
    at, size = CASES[where]
    cur[at] = base[at] + np.float32(size)
    b, c = torch.from_numpy(base).to(DEV), torch.from_numpy(cur).to(DEV)
    want = oracle.compress(base, cur, nbits)
    ws = lc.alloc_workspace(N, DEV)
    for options in (0, lc.OPT_NO_DEVICE_WAIT):
        s, tracked = lc.alloc_stream(N, nbits, DEV), b.clone()
        lc.compress_opt_async(tracked, c, nbits, s, ws, options, tracked)  # in place
        assert lc.last_status(ws) == 0
        assert to_np(s[: len(want)]).tobytes() == want.tobytes()
        assert np.array_equal(to_np(tracked).view(np.uint32), oracle.recover(base, [want]).view(np.uint32))
    assert lc.compress(b, c, nbits, workspace=ws).cpu().numpy().tobytes() == want.tobytes()
    check_update(lc, oracle, b, c, nbits, inplace=False)


def test_large_deltas_in_layers(lc, oracle):
    # the per-layer passes form keys of their own
    rng = np.random.default_rng(3)
    base = rng.normal(0, 0.02, N // 4 * 4).astype(np.float32)
    cur = base + rng.normal(0, 1e-3, base.size).astype(np.float32)
    cur[[5, 70_000]] += np.float32(3.0)
    seg = [0, 64, 50_000, 120_000, base.size]
    streams, off = lc.compress_segments(torch.from_numpy(base).to(DEV), torch.from_numpy(cur).to(DEV), seg, 4)
    for i in range(4):
        want = oracle.compress(base[seg[i]:seg[i + 1]], cur[seg[i]:seg[i + 1]], 4)
        assert to_np(streams[off[i]: off[i] + len(want)]).tobytes() == want.tobytes()
