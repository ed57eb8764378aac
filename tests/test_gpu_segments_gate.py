"""Per-layer compress: a layer of one chunk is prepared beside the statistics pass and writes only once all failures are known. Failures before, in and behind
such layers leave the right ones without a stream and without a tracked state, also where the state is advanced in place; and a layer of more tiles
than a look-back reads at once. Against the CPU oracle."""
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


SIZES = [64, 4096, 0, 5000, 1000, 70_000, 4, 4092, 9000, 8]


@pytest.mark.parametrize("bad", [None, 0, 1, 3, 4, 7, 9])  # segments with a non-finite delta: of one chunk and of several
def test_failures_around_small_layers(lc, oracle, bad):
    seg = np.concatenate([[0], np.cumsum(SIZES)]).tolist()
    rng = np.random.default_rng(7)
    base = rng.normal(0, 0.02, seg[-1]).astype(np.float32)
    cur = base + rng.normal(0, 1e-3, seg[-1]).astype(np.float32)
    if bad is not None:
        cur[seg[bad + 1] - 1] = np.inf
        cur[seg[-1] - 2] = np.nan  # and one in the last
    b, c = torch.from_numpy(base).to(DEV), torch.from_numpy(cur).to(DEV)
    off, total = lc.segments_layout(seg, 4)
    streams, ws = torch.full((total,), 7, dtype=torch.uint8, device=DEV), lc.alloc_workspace(max(SIZES), DEV)
    lc.compress_segments_async(b, c, seg, 4, streams, ws, b)  # in place
    assert lc.last_status(ws) == (lc.OK if bad is None else lc.ERR_NONFINITE)
    for i in range(len(SIZES)):
        got = to_np(streams[off[i]: off[i + 1]])
        if bad is not None and i >= bad:
            assert not got[:4].any()  # no stream
            assert np.array_equal(to_np(b[seg[i]: seg[i + 1]]).view(np.uint32), base[seg[i]: seg[i + 1]].view(np.uint32))
            continue
        want = oracle.compress(base[seg[i]: seg[i + 1]], cur[seg[i]: seg[i + 1]], 4)
        assert got[: len(want)].tobytes() == want.tobytes()
        after = oracle.recover(base[seg[i]: seg[i + 1]], [want])
        assert np.array_equal(to_np(b[seg[i]: seg[i + 1]]).view(np.uint32), after.view(np.uint32))


@pytest.mark.parametrize("tiles", [31, 33, 127, 128, 129, 260])
def test_layers_of_many_tiles(lc, oracle, tiles):
    n = tiles * 8 * 4096 - 4 * (tiles % 3)
    seg = [0, 100, 100 + n, 100 + n + 5000]
    rng = np.random.default_rng(tiles)
    base = rng.normal(0, 0.02, seg[-1]).astype(np.float32)
    cur = base + rng.normal(0, 1e-3, seg[-1]).astype(np.float32)
    streams, off = lc.compress_segments(torch.from_numpy(base).to(DEV), torch.from_numpy(cur).to(DEV), seg, 3)
    for i in range(3):
        want = oracle.compress(base[seg[i]: seg[i + 1]], cur[seg[i]: seg[i + 1]], 3)
        assert to_np(streams[off[i]: off[i] + len(want)]).tobytes() == want.tobytes()
