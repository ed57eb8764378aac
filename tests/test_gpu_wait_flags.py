"""A blocking call behind other work in the CUDA stream waits the way the device's flags say: with blocking synchronisation the thread sleeps.
A process per flag, since the flags belong to the device's primary context."""
import os
import subprocess
import sys

import pytest
import torch

from conftest import ROOT

pytestmark = pytest.mark.gpu

CHILD = """
import ctypes, sys, time
flags = int(sys.argv[1])
cuda = ctypes.CDLL("libcuda.so.1")
assert cuda.cuInit(0) == 0 and cuda.cuDevicePrimaryCtxSetFlags_v2(0, flags) == 0
import torch
from paper_2009_13003_b200 import binding
base = torch.randn(61_706, device="cuda:0")
cur = base * 1.01
work = torch.ones(1 << 28, device="cuda:0")
stream, workspace = binding.alloc_stream(base.numel(), 4, "cuda:0"), binding.alloc_workspace(base.numel(), "cuda:0")
want = binding.compress(base, cur, 4, stream, workspace).clone()
have, active = ctypes.c_uint(), ctypes.c_int()
assert cuda.cuDevicePrimaryCtxGetState(0, ctypes.byref(have), ctypes.byref(active)) == 0 and have.value & 7 == flags, have.value
wall = cpu = 0.0
for repeats in (0, 10, 100, 300):  # up to about 0.1 s of work in the stream ahead of the call
    for _ in range(repeats):
        work.neg_()
    t, c = time.perf_counter(), time.thread_time()
    got = binding.compress(base, cur, 4, stream, workspace)
    wall, cpu = time.perf_counter() - t, time.thread_time() - c
    assert torch.equal(got, want)
    out = binding.recover(base, [got])
print(wall, cpu)
"""


@pytest.mark.parametrize("flags", [0, 1, 2, 4])  # automatic, spin, yield, blocking
def test_the_wait_follows_the_flags_of_the_device(flags):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    done = subprocess.run([sys.executable, "-c", CHILD, str(flags)], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert done.returncode == 0, done.stderr
    wall, cpu = map(float, done.stdout.split())
    assert wall > 0.03  # the work that was queued
    if flags == 4:
        assert cpu < 0.25 * wall
