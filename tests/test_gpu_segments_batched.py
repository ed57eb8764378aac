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
