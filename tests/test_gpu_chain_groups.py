"""A chain of streams goes through in launches of one to four; however they are grouped, the state is the one that the streams
recover one at a time. Bit for bit.
"""
import pytest
import torch

from test_gpu_parity import DEV, make_case

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 5000, 40 * 4096 + 1, 3_000_001])
def test_groups_of_a_chain(n):
    from paper_2009_13003_b200 import binding as lc

    streams = []
    for j in range(lc.MAX_CHAIN):
        base, cur = make_case(n, 300 + 2 * j, dist="gauss" if j % 2 else "lognormal")
        streams.append(lc.compress(base, cur, 4).clone())
    want = base.clone()
    ws = lc.alloc_workspace(0, DEV)
    for k in range(1, lc.MAX_CHAIN + 1):
        want = lc.recover(want, streams[k - 1 : k], torch.empty_like(base), ws)
        got = lc.recover(base, streams[:k], torch.empty_like(base), ws)
        assert torch.equal(got.view(torch.int32), want.view(torch.int32)), k
