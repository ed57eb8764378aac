"""Calls that follow each other on one stream without a wait in between, sharing one workspace, and the same calls captured
in a CUDA graph: the kernels of a call may begin before the one ahead of them has ended, those of the next call may not.
Against the same calls made one by one.
"""
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


SIZES = [4096, 61_706, 140_000, 131_073, 1_000_003, 500, 3_000_000]


def jobs(lc):
    out = []
    for i, n in enumerate(SIZES):
        base, cur = make_case(n, 600 + i, dist=("lognormal", "gauss")[i % 2])
        nbits = 2 + i % 5
        begin = [0, n // 16 * 4, n // 8 * 4, n // 4 * 4]
        out.append((base, cur, nbits, torch.zeros(lc.stream_bound(n, nbits), dtype=torch.uint8, device=DEV), base.clone(),
                    torch.empty_like(base), begin, torch.zeros(lc.segments_layout(begin, nbits)[1], dtype=torch.uint8, device=DEV)))
    return out


def enqueue(lc, work, ws):
    for base, cur, nbits, stream, tracked, out, begin, streams in work:
        tracked.copy_(base)
        lc.compress_update_async(tracked, cur, nbits, stream, tracked, ws)
        lc.recover_async(base, [stream] * 5, out, ws)
        lc.compress_segments_async(base, cur, begin, nbits, streams, ws)
        lc.merge_async(base, [stream, stream], nbits, stream, out, ws)


def results(lc, work, ws, one_by_one):
    if one_by_one:
        for job in work:
            enqueue(lc, [job], ws)
            torch.cuda.synchronize()
    else:
        enqueue(lc, work, ws)
        torch.cuda.synchronize()
    return [t.clone() for job in work for t in (job[3], job[4], job[5], job[7])]


def test_back_to_back_and_captured(lc):
    ws = lc.alloc_workspace(max(SIZES), DEV)
    want = results(lc, jobs(lc), ws, one_by_one=True)
    work = jobs(lc)
    for _ in range(3):
        for job in work:
            job[3].zero_(), job[7].zero_()
        got = results(lc, work, ws, one_by_one=False)
        assert all(torch.equal(a.view(torch.uint8), b.view(torch.uint8)) for a, b in zip(want, got))
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        enqueue(lc, work, ws)
    for _ in range(3):
        for job in work:
            job[3].zero_(), job[5].zero_(), job[7].zero_()
        graph.replay()
        torch.cuda.synchronize()
        got = [t for job in work for t in (job[3], job[4], job[5], job[7])]
        assert all(torch.equal(a.view(torch.uint8), b.view(torch.uint8)) for a, b in zip(want, got))
