"""Chains of layers in every grouping, whose rule depends on nbits, and chains of three by either kernel, which the chunks' size decides.
The state is the one that the streams recover one at a time. Bit for bit.
"""
import numpy as np
import pytest
import torch

from test_gpu_leading_ones import deltas
from test_gpu_parity import DEV, assert_recover_parity

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nbits", [3, 4, 5, 9])
def test_groups_of_a_chain_of_layers(nbits):
    from paper_2009_13003_b200 import binding as lc, synth

    begin = np.cumsum([0, 4, 4096, 0, 33 * 4096 + 8, 1000, 70 * 4096]).tolist()
    base = synth.normal(begin[-1], 0.02, DEV, 1)
    cur, streams = base.clone(), []
    for j in range(lc.MAX_CHAIN):
        cur = cur + synth.sweep_delta("gauss" if j % 2 else "lognormal", begin[-1], DEV, 300 + j)
        streams.append(lc.compress_segments(base, cur, begin, nbits)[0].clone())
    want = base.clone()
    for k in range(1, lc.MAX_CHAIN + 1):
        want = lc.recover_segments(want, streams[k - 1 : k], begin, nbits)
        got = lc.recover_segments(base, streams[:k], begin, nbits)
        assert torch.equal(got.view(torch.int32), want.view(torch.int32)), k


@pytest.mark.parametrize("codes", [32, 36, 40, 90, 200])  # 5, 5.2 and 5.4 bits a code, where the kernel changes, and well above
def test_three_streams(oracle, codes):
    from paper_2009_13003_b200 import binding as lc

    n = 45 * 4096 + 2500
    base = torch.from_numpy(np.random.default_rng(9).standard_normal(n).astype(np.float32)).to(DEV)
    streams = [oracle.compress(np.zeros(n, np.float32), deltas([1] * codes, n, 20 + j), 8) for j in range(3)]
    assert_recover_parity(lc, oracle, base, streams)
    assert_recover_parity(lc, oracle, base, streams + streams[:2])
