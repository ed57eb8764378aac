"""Chunks that outgrow their columns or their image, which are coded again from the CTA's tables: stretches of rare exponents of several lengths in a vector of
frequent ones, at its beginning, over chunk edges and before its partial last chunk; streams and tracked states, flat and in layers, against the CPU oracle."""
import numpy as np
import pytest
import torch

from test_gpu_parity import DEV, to_np
from test_gpu_update import check_update

pytestmark = pytest.mark.gpu
N = 61 * 4096 + 500


@pytest.fixture(scope="module")
def lc():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2009_13003_b200 import binding

    binding.lib()
    return binding


@pytest.mark.parametrize("nbits", [2, 3, 4, 5, 6, 9])
@pytest.mark.parametrize("share", [4096, 8192 + 100, 300])  # elements of a stretch
def test_stretches_of_rare_exponents(lc, oracle, nbits, share):
    rng = np.random.default_rng(nbits * 7 + share)
    base = rng.normal(0, 0.02, N).astype(np.float32)
    delta = rng.choice([-1, 1], N) * 1.5e-3
    for at in (0, 9 * 4096 + 2000, 60 * 4096):
        m = min(share, N - at)
        delta[at: at + m] = rng.choice([-1, 1], m) * 1.3 * np.exp2(rng.integers(-12 if nbits > 4 else -9, 0, m))
    cur = base + delta.astype(np.float32)
    b, c = torch.from_numpy(base).to(DEV), torch.from_numpy(cur).to(DEV)
    check_update(lc, oracle, b, c, nbits, inplace=True)
    b = torch.from_numpy(base).to(DEV)
    stream = lc.compress(b, c, nbits)
    assert np.array_equal(to_np(lc.recover(b, [stream])).view(np.uint32), oracle.recover(base, [to_np(stream)]).view(np.uint32))
    seg = [0, 20_000, N // 4 * 4]
    streams, off = lc.compress_segments(b[: seg[-1]], c[: seg[-1]], seg, nbits)
    for i in range(2):
        want = oracle.compress(base[seg[i]: seg[i + 1]], cur[seg[i]: seg[i + 1]], nbits)
        assert to_np(streams[off[i]: off[i] + len(want)]).tobytes() == want.tobytes()
