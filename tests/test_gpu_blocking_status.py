"""The blocking calls of the binding look at the status word: a pass that reports an error raises, also when it has left a
stream with a header. The device reports nothing of the kind here; the word is set behind the pass, on the same CUDA stream.
"""
import ctypes as C
import threading

import numpy as np
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


@pytest.mark.parametrize("n", [1000, 61_706, 300_007])
def test_an_error_behind_a_complete_stream_raises(lc, monkeypatch, n):
    base, cur = make_case(n, 17)
    ws, cache = lc.alloc_workspace(n, DEV), lc.alloc_length_cache(DEV)
    good = lc.compress(base, cur, 4, None, ws).clone()

    def with_error(enqueue):
        def call(*args, **kw):
            enqueue(*args, **kw)
            ws[:4].view(torch.int32).fill_(lc.ERR_TIMEOUT)
        return call

    for name in ("compress_async", "compress_opt_async", "compress_update_async", "compress_cached_async", "merge_async", "recover_async"):
        monkeypatch.setattr(lc, name, with_error(getattr(lc, name)))
    for call in (lambda: lc.compress(base, cur, 4, None, ws), lambda: lc.compress(base, cur, 4, None, ws, mean=True),
                 lambda: lc.compress_update(base, cur, 4, workspace=ws), lambda: lc.compress_cached(base, cur, 4, cache, None, ws),
                 lambda: lc.merge(base, [good, good], 4, workspace=ws), lambda: lc.recover(base, [good], workspace=ws)):
        with pytest.raises(lc.LCError) as e:
            call()
        assert e.value.code == lc.ERR_TIMEOUT
    monkeypatch.undo()
    assert torch.equal(lc.compress(base, cur, 4, None, ws), good)


def test_wait_with_and_without_a_page(lc):
    n = 61_706
    base, cur = make_case(n, 18)
    ws = lc.alloc_workspace(n, DEV)
    s = lc.compress(base, cur, 3, None, ws)
    want = bytes(lc.stream_info(s))
    pinned, plain = torch.empty(128, dtype=torch.uint8, pin_memory=True), np.zeros(256, np.uint8)
    at = (plain.ctypes.data + 15) // 16 * 16  # ordinary memory: the call copies instead
    cs = lc._cs(torch.device(DEV))
    for page in (None, pinned.data_ptr(), at):
        for status in (lc.OK, lc.ERR_NONFINITE, lc.OK):
            ws[:4].view(torch.int32).fill_(status)
            info = lc.LCInfo()
            assert lc.lib().lc_wait(ws.data_ptr(), s.data_ptr(), C.byref(info), page, cs) == status
            assert bytes(info) == want
            assert lc.lib().lc_wait(ws.data_ptr(), None, None, page, cs) == status
    torch.cuda.synchronize()  # no error is left behind


def test_first_call_of_a_thread_under_a_default_device(lc):
    base, cur = make_case(5000, 19)
    want, got = lc.compress(base, cur, 4), []

    def work():
        with torch.device(DEV):
            got.append(lc.compress(base, cur, 4))
        torch.cuda.synchronize()

    torch.cuda.synchronize()
    t = threading.Thread(target=work)
    t.start()
    t.join()
    assert len(got) == 1 and torch.equal(got[0], want)
