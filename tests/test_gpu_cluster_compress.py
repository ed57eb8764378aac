"""Vectors of 2 to 32 chunks, which one cluster of CTAs compresses in one launch, against the CPU oracle (and one chunk
more, which takes the general path). Bar: byte-identical streams, bit-identical tracked states.
"""
import pytest
import torch

from test_gpu_parity import DEV, _fibonacci_case, assert_stream_parity, make_case, to_np
from test_gpu_update import check_update

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lc():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2009_13003_b200 import binding

    binding.lib()
    return binding


# one element into, and the whole of, the last chunk of each cluster size: 2, 4, 8, 16 CTAs, then two chunks per CTA
@pytest.mark.parametrize("chunks", [1, 2, 3, 4, 5, 8, 9, 16, 17, 31, 32, 33])
@pytest.mark.parametrize("last", [1, 4096])
def test_cluster_sizes(lc, oracle, chunks, last):
    n = (chunks - 1) * 4096 + last
    for dist, nbits in (("lognormal", 9), ("gauss", 3)):
        base, cur = make_case(n, chunks * 10 + nbits, dist=dist)
        assert_stream_parity(lc, oracle, base, cur, nbits)
        check_update(lc, oracle, base, cur, nbits, inplace=True)


@pytest.mark.parametrize("front", [False, True])
def test_chunk_larger_than_its_image(lc, oracle, front):
    # rare symbols together in one chunk: up to 25 bits an element there, about two on average
    base, cur = _fibonacci_case(22, False)
    rare, _ = torch.sort(cur, descending=True)
    few, many = rare[:4096], torch.full((120_000,), float(rare[-1]), device=DEV)
    cur = torch.cat([few, many] if front else [many[:60_001], few, many[60_001:]])
    check_update(lc, oracle, torch.zeros_like(cur), cur, 9, inplace=False)


def test_failure_and_large_deltas(lc, oracle):
    base, cur = make_case(50_000, 9)
    bad = cur.clone()
    bad[33_333] = float("inf")
    stream, ws, keep = lc.alloc_stream(50_000, 4, DEV), lc.alloc_workspace(50_000, DEV), base.clone()
    lc.compress_update_async(keep, bad, 4, stream, keep, ws)
    assert lc.last_status(ws) == lc.ERR_NONFINITE and lc.stream_info(stream).valid == 0
    assert torch.equal(keep, base)
    cur[::97] += 1e4  # exponent fields >= 128
    check_update(lc, oracle, base, cur, 6, inplace=True)
    assert to_np(cur).size == 50_000
