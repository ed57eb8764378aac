"""lc_stream_info and lc_last_status take any device address: a header at an odd offset of a packed buffer, and memory of
a device that is not the current one (skipped where fewer than two devices are visible).
"""
import threading

import pytest
import torch

from test_gpu_parity import DEV, make_case

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lc():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2009_13003_b200 import binding

    binding.lib()
    return binding


@pytest.mark.parametrize("offset", [1, 2, 3, 4, 7, 16])
def test_header_at_any_offset(lc, offset):
    n, nbits = 61_706, 3
    base, cur = make_case(n, 41)
    s = lc.compress(base, cur, nbits)
    packed = torch.full((offset + s.numel(),), 0xFF, dtype=torch.uint8, device=DEV)
    packed[offset:] = s
    want, got = lc.stream_info(s), lc.stream_info(packed[offset:])
    assert got.valid == 1 and got.n == n and got.total_bytes == s.numel()
    assert bytes(want) == bytes(got)
    assert lc.stream_info(packed).valid == 0


def test_threads_with_streams_of_their_own(lc):
    base, cur = make_case(4096, 42)
    seen = []

    def work():
        with torch.cuda.stream(torch.cuda.Stream()):
            ws = lc.alloc_workspace(4096, DEV)
            s = lc.compress(base, cur, 4, None, ws)
            seen.append((lc.last_status(ws), lc.stream_info(s).total_bytes == s.numel()))

    torch.cuda.synchronize()
    threads = [threading.Thread(target=work) for _ in range(8)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert seen == [(lc.OK, True)] * 8


def test_memory_of_another_device(lc):
    if torch.cuda.device_count() < 2:
        pytest.skip("needs two CUDA devices")
    with torch.cuda.device(1):
        base = torch.randn(10_000, device="cuda:1")
        ws = lc.alloc_workspace(10_000, "cuda:1")
        s = lc.compress(base, base * 1.01, 4, None, ws)
        torch.cuda.synchronize()
    with torch.cuda.device(0):
        assert lc.last_status(ws) == lc.OK and lc.stream_info(s).total_bytes == s.numel()
