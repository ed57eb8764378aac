"""The encoder's table of pairs at its limits: how many plane-byte values (exponents of both signs) the kept buckets span,
elements outside the span that the table covers, and codes too long for a pair. Against the CPU oracle, byte for byte.
"""
import pytest
import torch

from test_gpu_parity import DEV, assert_stream_parity
from test_gpu_update import check_update

pytestmark = pytest.mark.gpu

N = 40 * 4096 + 13  # more chunks than the single-launch path takes


@pytest.fixture(scope="module")
def lc():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2009_13003_b200 import binding

    binding.lib()
    return binding


def deltas(weights, seed):
    """N deltas; weights: {(sign, exponent field): share}."""
    g = torch.Generator(device="cpu").manual_seed(seed)
    keys = list(weights)
    pick = torch.multinomial(torch.tensor([float(weights[k]) for k in keys]), N, replacement=True, generator=g)
    pick[: len(keys)] = torch.arange(len(keys))  # every bucket occurs
    head = torch.tensor([(s << 31 | e << 23) - (1 << 32 if s else 0) for s, e in keys], dtype=torch.int32)
    bits = head[pick] | torch.randint(0, 1 << 23, (N,), generator=g, dtype=torch.int32)
    return bits.view(torch.float32)[torch.randperm(N, generator=g)].to(DEV)


@pytest.mark.parametrize("span", [1, 2, 29, 30, 31, 32, 33, 34, 60])
@pytest.mark.parametrize("nbits", [4, 5, 6, 9])
def test_spans(lc, oracle, span, nbits):
    # `span` neighbouring plane bytes, most elements in the middle
    w = {(b & 1, b >> 1): 2.0 ** -abs(i - span // 2) for i, b in enumerate(range(200 - span, 200))}
    d = deltas(w, span)
    check_update(lc, oracle, torch.zeros_like(d), d, nbits, inplace=False)
    assert_stream_parity(lc, oracle, torch.zeros_like(d), d, nbits)


@pytest.mark.parametrize("rare", [1e-9, 1e-3, 0.02, 0.3])
@pytest.mark.parametrize("where", ["above", "below", "both", "edges"])
def test_elements_outside_the_table(lc, oracle, rare, where):
    w = {(s, e): 1.0 for s in (0, 1) for e in range(100, 106)}
    if where in ("above", "both"):
        w.update({(0, 127): rare, (1, 125): rare})
    if where in ("below", "both"):
        w.update({(0, 40): rare, (1, 1): rare, (0, 1): rare, (0, 0): rare})
    if where == "edges":  # both ends of the byte range
        w = {(1, 127): 1.0, (0, 127): 0.5, (0, 1): 1.0, (1, 1): rare, (1, 0): 0.2}
    d = deltas(w, 7)
    for nbits in (3, 9):
        check_update(lc, oracle, torch.zeros_like(d), d, nbits, inplace=False)


def test_pairs_longer_than_an_entry(lc, oracle):
    # neighbouring rare symbols of 13 to 16 bits each, in runs
    w = {(i & 1, 110 - i // 2): 2.0 ** -i for i in range(17)}
    d = deltas(w, 3)
    rare, _ = torch.sort(d.abs())
    d[4096:4096 + 600] = rare[:600]
    check_update(lc, oracle, torch.zeros_like(d), d, 5, inplace=False)
