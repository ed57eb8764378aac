"""The index of the decoder's table by leading ones, restated in numpy's float32: every window of 15 bits falls into the
entry whose range of complements it lies in, at the smallest and largest value of each entry included. CPU only; the
kernel's own form is compared with the oracle in test_gpu_leading_ones.py.
"""
import numpy as np


def entry_range(i):
    e, q = i // 8, i % 8  # the exponent plus one, the three bits behind the leading one of the complement
    least, end = ((8 + q) << e) >> 4, ((9 + q) << e) >> 4
    return least, max(least, end - 1)


def index_of(window):
    x = (np.uint32(0x3F800000) | window.astype(np.uint32)).view(np.float32)
    # fp32 fused multiply-add: the product and the sum are exact in 64 bits (24 + 24 bits, and exponents of 0 and -24)
    f = (x.astype(np.float64) * -(1.0 - 2.0 ** -24) + (1.0 + 32767 * 2.0 ** -23)).astype(np.float32)
    return (f.view(np.uint32) >> 20).astype(np.int64) - (127 - 24) * 8


def test_every_window_falls_into_its_entry():
    w = np.arange(1 << 15)
    i = index_of(w)
    assert i.min() >= 0 and i.max() == 127
    least, most = np.array([entry_range(k) for k in range(128)]).T
    v = 32767 - w
    assert np.all(least[i] <= v) and np.all(v <= most[i])
    # entries of eight windows or more are met by all of them, so an entry with one code holds it for all its windows
    for k in range(32, 128):
        assert (i == k).sum() == most[k] - least[k] + 1
    # and below that a window has one entry to itself
    for k in range(32):
        assert (i == k).sum() <= 1
