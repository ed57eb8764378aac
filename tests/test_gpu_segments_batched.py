"""Per-layer calls over more segments than one launch takes, with empty, tiny, ragged and large segments, against the CPU
oracle segment by segment. Bar: byte-identical streams, bit-identical states; of several failures the first segment's.
"""
import random

import numpy as np
import pytest
import torch

from test_gpu_parity import DEV, to_np
from test_gpu_segments import layered_case

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lc():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2009_13003_b200 import binding

    binding.lib()
    return binding


def many_sizes(nseg, seed):
    rng = random.Random(seed)
    return [rng.choice([0, 4, 64, 1000, 4092, 4096, 4100, 9408, 36864, 4 * rng.randint(1, 30000)]) for _ in range(nseg)]


@pytest.mark.parametrize("nseg,nbits,chain", [(1, 4, 1), (40, 4, 5), (161, 3, 2), (400, 6, 1)])
def test_many_segments(lc, oracle, nseg, nbits, chain):
    sizes = many_sizes(nseg, nseg + nbits)
    base, curs, begin = layered_case(sizes, 900 + nseg, chain)
    offsets, total = lc.segments_layout(begin, nbits)
    host, tracked, bufs = to_np(base).copy(), base.clone(), []
    for t, cur in enumerate(curs):
        streams = torch.full((total,), 0xA5, dtype=torch.uint8, device=DEV)
        lc.compress_segments(tracked, cur, begin, nbits, streams=streams, tracked_out=tracked)
        got, ch = to_np(streams), to_np(cur)
        for i, (a, b) in enumerate(zip(begin[:-1], begin[1:])):
            want = oracle.compress(host[a:b], ch[a:b], nbits)
            assert got[offsets[i]: offsets[i] + want.size].tobytes() == want.tobytes(), "segment %d of %d" % (i, b - a)
            assert (got[offsets[i] + lc.stream_bound(b - a, nbits): offsets[i + 1]] == 0xA5).all(), "wrote past its slot"
            host[a:b] = oracle.recover(host[a:b], [want])
        assert np.array_equal(to_np(tracked).view(np.uint32), host.view(np.uint32)), "tracked state"
        bufs.append(streams)
    out = lc.recover_segments(base, bufs, begin, nbits)
    assert np.array_equal(to_np(out).view(np.uint32), host.view(np.uint32)), "recovered state"
    x = base.clone()
    lc.recover_segments(x, bufs, begin, nbits, out=x)
    assert torch.equal(x, out)


def test_first_of_several_damaged_segments_is_reported(lc):
    sizes = [4096] * 30
    base, curs, begin = layered_case(sizes, 31, 1)
    streams, off = lc.compress_segments(base, curs[0], begin, 4)
    ws = lc.alloc_workspace(0, DEV)
    for first, second in ((7, 8), (8, 7), (0, 29)):
        bad = streams.clone()
        bad[off[first]] = 0                                    # no magic: LC_ERR_FORMAT
        bad[off[second] + 8: off[second] + 10] = 1             # another n: LC_ERR_MISMATCH
        lc.recover_segments_async(base, [streams, bad], begin, 4, torch.empty_like(base), ws)
        assert lc.last_status(ws) == (lc.ERR_FORMAT if first < second else lc.ERR_MISMATCH)
    # the damaged stream of a later group of four counts after every stream of the first group, of the same segment
    bad = streams.clone()
    bad[off[3]] = 0
    worse = streams.clone()
    worse[off[3] + 8: off[3] + 10] = 1
    lc.recover_segments_async(base, [streams, bad, streams, streams, worse], begin, 4, torch.empty_like(base), ws)
    assert lc.last_status(ws) == lc.ERR_FORMAT


def check_segments(lc, oracle, base, cur, begin, nbits):
    """In place, against the oracle segment by segment."""
    offsets, total = lc.segments_layout(begin, nbits)
    bh, ch = to_np(base).copy(), to_np(cur)
    tracked = base.clone()
    streams = torch.full((total,), 0xA5, dtype=torch.uint8, device=DEV)
    longest = max(b - a for a, b in zip(begin[:-1], begin[1:]))
    wsb = lc.workspace_bytes(longest)  # no more than the call asks for: groups end where it is full
    ws = torch.full((wsb + 256,), 0x5A, dtype=torch.uint8, device=DEV)
    lc.compress_segments(tracked, cur, begin, nbits, streams=streams, workspace=ws[:wsb], tracked_out=tracked)
    assert bool((ws[wsb:] == 0x5A).all()), "wrote past the workspace"
    got, state = to_np(streams), to_np(tracked)
    for i, (a, b) in enumerate(zip(begin[:-1], begin[1:])):
        want = oracle.compress(bh[a:b], ch[a:b], nbits)
        assert got[offsets[i]: offsets[i] + want.size].tobytes() == want.tobytes(), "segment %d of %d" % (i, b - a)
        assert np.array_equal(state[a:b].view(np.uint32), oracle.recover(bh[a:b], [want]).view(np.uint32)), "segment %d" % i


def to_begin(sizes):
    return [int(v) for v in np.concatenate([[0], np.cumsum(sizes)])]


@pytest.mark.parametrize("nbits", [1, 4, 8, 9])
def test_segments_of_every_kind(lc, oracle, nbits):
    """Exponents the key plane does not hold, codes beyond 16 and 32 bits, entropy beyond a lane's column."""
    g = torch.Generator(device="cpu").manual_seed(nbits)

    def exponents(n, lo, hi):  # every (sign, exponent) of the range equally often: the longest streams
        e = torch.randint(lo, hi, (n,), generator=g, dtype=torch.int32)
        m = torch.randint(0, 1 << 23, (n,), generator=g, dtype=torch.int32)
        s = torch.randint(0, 2, (n,), generator=g, dtype=torch.int32)
        return ((s << 31) | (e << 23) | m).view(torch.float32)

    def fibonacci(k):
        from test_gpu_parity import _fibonacci_case

        x = _fibonacci_case(k, False)[1].cpu() * 2.0 ** -20
        return x[: x.numel() // 4 * 4]

    parts = [exponents(70_000, 1, 127), fibonacci(24), torch.zeros(50_000), exponents(4096, 1, 254), exponents(70_004, 60, 200),
             torch.cat([exponents(36_000, 1, 127), torch.full((300_000,), 1e-3)]), fibonacci(26), exponents(8, 100, 127)]
    cur = torch.cat(parts).to(DEV)
    check_segments(lc, oracle, torch.zeros_like(cur), cur, to_begin([p.numel() for p in parts]), nbits)


def test_groups_that_the_workspace_limits(lc, oracle):
    # many segments just above one chunk: a workspace for one of them holds the blocks of a dozen
    sizes = [4100, 4096, 8192, 4, 6000] * 40
    base, curs, begin = layered_case(sizes, 4100, 1)
    check_segments(lc, oracle, base, curs[0], begin, 5)


@pytest.mark.parametrize("failed", [0, 2, 3, 150, 199])
def test_segments_behind_a_failure_have_no_stream(lc, oracle, failed):
    sizes = [4096, 40_000, 1000, 12_292] * 50
    base, curs, begin = layered_case(sizes, 5, 1)
    cur, nbits = curs[0].clone(), 4
    for f in (failed, min(failed + 3, len(sizes) - 1)):
        cur[begin[f] + 7] = float("nan")
    offsets, total = lc.segments_layout(begin, nbits)
    ws = lc.alloc_workspace(max(sizes), DEV)
    tracked = base.clone()
    streams, _ = lc.compress_segments(base, curs[0], begin, nbits)  # valid streams of another call stand there
    good = to_np(streams).copy()
    lc.compress_segments_async(tracked, cur, begin, nbits, streams, ws, tracked)
    assert lc.last_status(ws) == lc.ERR_NONFINITE
    got = to_np(streams)
    for i in range(len(sizes)):
        if i < failed:
            assert got[offsets[i]: offsets[i] + 64].tobytes() == good[offsets[i]: offsets[i] + 64].tobytes()
        else:
            assert lc.stream_info(streams[offsets[i]:]).valid == 0
    assert torch.equal(tracked[begin[failed]:], base[begin[failed]:])
    if failed:
        want = lc.recover_segments(base[: begin[failed]].contiguous(), [streams], begin[: failed + 1], nbits)
        assert torch.equal(tracked[: begin[failed]], want)
