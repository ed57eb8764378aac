"""The scan of the encode pass over words that sum up groups of 256 chunks: streams around the edges of a tile, of a group and of the
64 groups that a look-back reads at once equal those of the two-pass scan, which looks nowhere back, and, where they are small, the oracle's."""
import pytest
import torch

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
CHUNK, GROUP = 4096, 256 * 4096


@pytest.fixture(scope="module")
def lc():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2009_13003_b200 import binding

    binding.lib()
    return binding


@pytest.mark.parametrize("nbits,fixed", [(4, False), (9, True)])  # eight warps a tile code, and four
@pytest.mark.parametrize("n", [33 * CHUNK, 40 * CHUNK + 1, GROUP - CHUNK, GROUP - 1, GROUP, GROUP + 1, GROUP + 9 * CHUNK + 77,
                               64 * GROUP, 65 * GROUP + 3, 130 * GROUP + 5 * CHUNK - 1])
def test_stream_at_group_edges(lc, oracle, n, nbits, fixed):
    from paper_2009_13003_b200 import synth

    base = synth.normal(n, 0.02, DEV, 5)
    cur = base + synth.lognormal_signed(n, 1e-4, 1.5, DEV, 6)
    ws = lc.alloc_workspace(n, DEV)
    got, want = lc.alloc_stream(n, nbits, DEV), lc.alloc_stream(n, nbits, DEV)
    options = lc.OPT_FIXED_WIDTH if fixed else 0
    lc.compress_opt_async(base, cur, nbits, want, ws, options | lc.OPT_NO_DEVICE_WAIT)
    assert lc.last_status(ws) == 0
    size = lc.stream_info(want).total_bytes
    for _ in range(3):
        got.zero_()
        lc.compress_opt_async(base, cur, nbits, got, ws, options)
        assert lc.last_status(ws) == 0
        assert torch.equal(got[:size], want[:size])
    if n <= 2 * GROUP and not fixed:
        assert got[:size].cpu().numpy().tobytes() == oracle.compress(base.cpu().numpy(), cur.cpu().numpy(), nbits).tobytes()
    tracked = torch.empty_like(base)
    lc.compress_opt_async(base, cur, nbits, got, ws, options, tracked)
    assert lc.last_status(ws) == 0 and torch.equal(got[:size], want[:size])
    assert torch.equal(tracked, lc.recover(base, [want[:size]]))
