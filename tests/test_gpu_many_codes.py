"""Recovery around the number of codes from which on a launch takes the two-level table without filling the other (128), alone and
beside streams of few codes. Against the CPU oracle, bit for bit.
"""
import numpy as np
import pytest
import torch

from test_gpu_leading_ones import deltas
from test_gpu_parity import DEV, assert_recover_parity

pytestmark = pytest.mark.gpu


def stream(oracle, codes, n, seed, fixed=False):
    return oracle.compress(np.zeros(n, np.float32), deltas([1] * codes, n, seed), 8, fixed=fixed)


@pytest.mark.parametrize("codes", [127, 128, 129, 130, 200])
@pytest.mark.parametrize("n", [4096, 20 * 4096 + 77])
def test_number_of_codes(oracle, codes, n):
    from paper_2009_13003_b200 import binding as lc

    base = torch.from_numpy(np.random.default_rng(9).standard_normal(n).astype(np.float32)).to(DEV)
    many = [stream(oracle, codes, n, 80 + j) for j in range(4)]
    for k in (1, 2, 3, 4):
        assert_recover_parity(lc, oracle, base, many[:k], inplace=k % 2 == 0)
    few = stream(oracle, 9, n, 90)
    for chain in ([few, many[0]], [many[0], few, few], [few, few, few, many[0]], [stream(oracle, codes, n, 91, fixed=True), many[0]]):
        assert_recover_parity(lc, oracle, base, chain)
