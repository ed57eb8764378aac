"""The bounded wait of the encode pass's scan over group words runs out: tile 0 is never coded, so its group never gets complete and the tiles of all later
groups meet an unfinished or aborted group word. Two groups, several, and more than the 64 that a look-back reads at once; with eight warps a tile and
with four; with and without the tracked state. Every wait is bounded; a normal call on the same workspace is complete again."""
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


def make(n, warps):
    from paper_2009_13003_b200 import synth

    if warps == 8:
        base = synth.normal(n, 0.02, DEV, 5)
        return base, base + synth.lognormal_signed(n, 1e-4, 1.5, DEV, 6), 4
    g = torch.Generator(device=DEV).manual_seed(7)  # some 230 buckets of about the same size: 7.8 bits an element
    exponent = torch.randint(-118, -2, (n,), device=DEV, generator=g)
    cur = torch.ldexp(torch.rand(n, device=DEV, generator=g) + 1.0, exponent)
    cur[::2].neg_()
    return torch.zeros(n, device=DEV), cur, 9


@pytest.mark.parametrize("warps", [8, 4])
@pytest.mark.parametrize("n", [GROUP + 9 * CHUNK + 77, 5 * GROUP, 66 * GROUP + 3 * CHUNK + 1])
def test_the_wait_runs_out_across_groups(lc, n, warps):
    base, cur, nbits = make(n, warps)
    ws, stream, want = lc.alloc_workspace(n, DEV), lc.alloc_stream(n, nbits, DEV), lc.alloc_stream(n, nbits, DEV)
    tracked = torch.empty_like(base)
    lc.compress_opt_async(base, cur, nbits, want, ws, lc.OPT_NO_DEVICE_WAIT)
    assert lc.last_status(ws) == lc.OK
    info = lc.stream_info(want)
    average = info.payload_bits // 8 // info.nchunks
    assert (average + average // 7 + 64 > 3072) == (warps == 4)  # half of a warp's share of 48 KB
    want = want[: info.total_bytes]
    state = lc.recover(base, [want])
    for spin_limit in (0, 300):
        lc.debug_compress_wait(base, cur, nbits, stream, ws, spin_limit, 1)
        assert lc.last_status(ws) == lc.ERR_TIMEOUT
        stream.zero_()
        assert torch.equal(lc.compress(base, cur, nbits, stream, ws), want)
        lc.debug_update_wait(base, cur, nbits, stream, tracked, ws, spin_limit, 1)
        assert lc.last_status(ws) == lc.ERR_TIMEOUT
        stream.zero_()
        got, tracked = lc.compress_update(base, cur, nbits, tracked, stream, ws)
        assert torch.equal(got, want) and torch.equal(tracked, state)
