"""A process that asked CUDA for blocking waits does not spend a core on a solve's wait for
its convergence reports. In a process of its own (the flag belongs to the device's primary
context): iterations of milliseconds (FP64 source iteration, 128,000 columns at N = 128: at
least 2 G FP64 FMAs each, over 1 ms at this GPU's rate), of which the host's launches (three, at
most 20 us each) and polls (at most a tenth of the time) take less than half by far; a
spinning wait would take all of it.
"""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

CODE = """
import ctypes, sys, time
sys.path.insert(0, %r)
cu = ctypes.CDLL("libcuda.so.1")
assert cu.cuInit(0) == 0 and cu.cuDevicePrimaryCtxSetFlags_v2(0, 4) == 0  # CU_CTX_SCHED_BLOCKING_SYNC
import torch
import __graft_entry__ as g
g.build()
from paper_1907_13013_gb300 import binding, inputs
p = inputs.random_slab(2000, 128, 127, seed=1, kernel="hg", thick=(2, 60), c=(0.7, 0.99), nrhs=32)
ctx = binding.context_for(p, precision="fp64")
out = torch.zeros((32, 2000, 2, 128), dtype=torch.float64, device="cuda")
ctx.solve("si", tol=0.0, max_iterations=3, out=out, raise_on_notconv=False)
t, c = time.perf_counter(), time.thread_time()
ctx.solve("si", tol=0.0, max_iterations=100, out=out, raise_on_notconv=False)
print("SHARE", (time.thread_time() - c) / (time.perf_counter() - t))
"""


def test_blocking_wait_sleeps():
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", CODE % root], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
    assert float(r.stdout.split("SHARE")[1]) < 0.5
