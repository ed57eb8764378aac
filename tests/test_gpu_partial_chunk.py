"""The vector's partial last chunk, which is coded and decoded four slots at a time with the slots beyond the end masked,
and the per-CTA preparation of the decode tables, against the CPU oracle. Bar: byte-identical streams, bit-identical states.
"""
import numpy as np
import pytest
import torch

from test_gpu_parity import DEV, _fibonacci_case, assert_recover_parity, make_case, to_np
from test_gpu_update import check_update

pytestmark = pytest.mark.gpu

# remainders at the edges of a slot group (4), of a step (128) and of the four steps that are read at once (512)
REMAINDERS = [1, 2, 3, 4, 5, 127, 128, 129, 130, 511, 512, 513, 4093, 4095]


@pytest.fixture(scope="module")
def lc():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2009_13003_b200 import binding

    binding.lib()
    return binding


@pytest.mark.parametrize("rem", REMAINDERS)
@pytest.mark.parametrize("dist,nbits", [("lognormal", 6), ("gauss", 2)])
def test_partial_chunk(lc, oracle, rem, dist, nbits):
    base, cur = make_case(2 * 4096 + rem, 500 + rem, dist=dist)
    stream = check_update(lc, oracle, base, cur, nbits, inplace=True)
    base, _ = make_case(2 * 4096 + rem, 500 + rem, dist=dist)
    for k in (1, 2, 4):
        assert_recover_parity(lc, oracle, base, [stream] * k)


@pytest.mark.parametrize("nsyms", [16, 20, 24])
@pytest.mark.parametrize("cut", [0, 1, 130, 2000])
def test_long_codes_in_the_partial_chunk(lc, oracle, nsyms, cut):
    # Fibonacci counts: codes of up to nsyms - 1 bits, i.e. longer than 16; the rare symbols stand at the vector's end
    base, cur = _fibonacci_case(nsyms, True)
    cur = (cur * 2.0 ** -20).flip(0)[cut:].clone()  # every |delta| < 2: the key plane identifies the buckets
    base = torch.zeros_like(cur)
    stream = check_update(lc, oracle, base, cur, 5, inplace=False)
    assert_recover_parity(lc, oracle, base, [stream])
    assert_recover_parity(lc, oracle, base, [stream] * 3)


def test_streams_of_every_kind_in_one_chain(lc, oracle):
    n = 5 * 4096 + 77
    base, cur = make_case(n, 77, dist="lognormal")
    wide = base + torch.randn(n, device=DEV) * torch.exp2(torch.randint(-100, 100, (n,), device=DEV).float())
    zero = base.clone()
    streams = [
        lc.compress(base, wide, 9),              # hundreds of symbols: several blocks of 32
        lc.compress(base, cur, 5, fixed=True),   # an incomplete code
        lc.compress(base, zero, 3),              # a single symbol: no payload
        lc.compress(base, cur, 8, mean=True),
        lc.compress(base, cur, 1),
    ]
    host = [to_np(s) for s in streams]
    for k in range(1, len(host) + 1):
        assert_recover_parity(lc, oracle, base, host[:k])
    assert_recover_parity(lc, oracle, base, host[::-1], inplace=True)
