"""Per-layer compress with layers so large that they go through the passes for one vector, between small ones, empty ones
and ones of many chunks. Bar: the streams that the slices give by themselves (one of them against the CPU oracle too), the
state that they recover, and no stream behind a segment that failed, whichever way it and the others go.
"""
import numpy as np
import pytest
import torch

from test_gpu_parity import DEV, ORACLE_THREADS, to_np

pytestmark = pytest.mark.gpu

# beyond the line of a call without a tracked state, and beyond that of any call
LARGE, LARGER = (40 << 20) + 4, (64 << 20) + 3 * 4096 + 8
SIZES = [1000, LARGER, 9408, 0, 300_000, LARGE, LARGER + 4096, 0, 64, 20_480]


@pytest.fixture(scope="module")
def lc():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2009_13003_b200 import binding

    binding.lib()
    return binding


@pytest.fixture(scope="module")
def case():
    from paper_2009_13003_b200 import synth

    begin = [0]
    for s in SIZES:
        begin.append(begin[-1] + s)
    base = synth.normal(begin[-1], 0.02, DEV, 51)
    return base, base + synth.sweep_delta("lognormal", begin[-1], DEV, 52), begin


@pytest.mark.parametrize("tracked", ["none", "apart", "in place"])
def test_streams_of_the_slices(lc, oracle, case, tracked):
    base, cur, begin = case
    nbits = 4
    offsets, total = lc.segments_layout(begin, nbits)
    streams = torch.full((total,), 0xA5, dtype=torch.uint8, device=DEV)
    ws = lc.alloc_workspace(max(SIZES), DEV)
    ws.fill_(0x5A)
    x = base.clone()
    out = {"none": None, "apart": torch.empty_like(base), "in place": x}[tracked]
    lc.compress_segments(x, cur, begin, nbits, streams, ws, out)
    for i, (a, b) in enumerate(zip(begin[:-1], begin[1:])):
        want = lc.compress(base[a:b], cur[a:b], nbits)
        assert torch.equal(streams[offsets[i]: offsets[i] + want.numel()], want), "segment %d" % i
        assert bool((streams[offsets[i] + lc.stream_bound(b - a, nbits): offsets[i + 1]] == 0xA5).all())
        if out is not None and b > a:
            assert torch.equal(out[a:b], lc.recover(base[a:b], [want])), "tracked state of segment %d" % i
    if tracked == "none":
        a, b = begin[1], begin[2]
        want = oracle.compress(to_np(base[a:b]), to_np(cur[a:b]), nbits, threads=ORACLE_THREADS)
        assert to_np(streams[offsets[1]: offsets[1] + want.size]).tobytes() == want.tobytes()


@pytest.mark.parametrize("failed", [(0,), (1,), (2,), (4,), (5,), (6,), (8,), (9,), (6, 1), (9, 5), (2, 6)])
def test_no_stream_behind_a_failed_segment(lc, case, failed):
    base, cur, begin = case
    bad = cur.clone()
    for i in failed:
        bad[begin[i + 1] - 1] = float("inf")
    offsets, total = lc.segments_layout(begin, 4)
    streams = torch.full((total,), 0xA5, dtype=torch.uint8, device=DEV)
    ws = lc.alloc_workspace(max(SIZES), DEV)
    for _ in range(2):  # the second call must not remember the first
        lc.compress_segments_async(base, bad, begin, 4, streams, ws)
        assert lc.last_status(ws) == lc.ERR_NONFINITE
        for i in range(len(SIZES)):
            assert lc.stream_info(streams[offsets[i]:]).valid == (1 if i < min(failed) else 0), "segment %d" % i
    lc.compress_segments(base, cur, begin, 4, streams, ws)
    assert all(lc.stream_info(streams[offsets[i]:]).valid == 1 for i in range(len(SIZES)))


def test_empty_segments_take_any_tracked_state(lc):
    # nothing is written, so the address is not looked at, as in lc_compress_update of an empty vector
    base = torch.zeros(16, device=DEV)
    begin = [0, 0, 0]
    streams, off = lc.compress_segments(base[:0], base[:0], begin, 4, tracked_out=base[1:])
    assert all(lc.stream_info(streams[o:]).valid == 1 for o in off[:-1])
