"""Recovery of a vector of at most 32 chunks clears the status word in its own launch: whatever the workspace held before, results and errors are those of any
other call. Sizes on both sides of that line and of a CTA's four chunks, chains of one and two launches, damaged streams. Against the CPU oracle."""
import numpy as np
import pytest
import torch

from test_gpu_parity import DEV, make_case, to_np

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lc():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2009_13003_b200 import binding

    binding.lib()
    return binding


@pytest.mark.parametrize("k", [1, 2, 3, 4, 5, 8])
@pytest.mark.parametrize("n", [1, 4096, 4 * 4096 + 1, 17 * 4096, 32 * 4096, 32 * 4096 + 1])
def test_status_is_cleared(lc, oracle, n, k):
    base, cur = make_case(n, n % 1000 + k)
    stream = lc.compress(base, cur, 4)
    want = oracle.recover(to_np(base), [to_np(stream)] * k)
    ws, out = lc.alloc_workspace(0, DEV), torch.empty_like(base)
    for stale in (0, 255, 127):
        ws.fill_(stale)
        lc.recover_async(base, [stream] * k, out, ws)
        assert lc.last_status(ws) == lc.OK
        assert np.array_equal(to_np(out).view(np.uint32), want.view(np.uint32))
    bad = stream.clone()
    bad[0] ^= 1  # the magic
    other = lc.compress(*make_case(n + 4, 1), 4)  # another number of elements
    for at in range(k):
        for damaged, code in ((bad, lc.ERR_FORMAT), (other, lc.ERR_MISMATCH)):
            chain = [stream] * k
            chain[at] = damaged
            if at + 1 < k:
                chain[at + 1] = bad if damaged is other else other  # the first failure of a launch stays
            lc.recover_async(base, chain, out, ws)
            assert lc.last_status(ws) == code
    chunk_index = 64 + 16 * lc.stream_info(stream).nsym
    broken = stream.clone()
    broken[chunk_index: chunk_index + 8].view(torch.int64).fill_(16)  # the first chunk begins behind the payload's beginning
    lc.recover_async(base, [broken] * k, out, ws)
    assert lc.last_status(ws) == lc.ERR_FORMAT
    lc.recover_async(base, [stream] * k, out, ws)
    assert lc.last_status(ws) == lc.OK and np.array_equal(to_np(out).view(np.uint32), want.view(np.uint32))
