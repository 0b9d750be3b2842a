"""A process that asked CUDA for blocking synchronisation keeps its host core while a solve runs: the thread sleeps
until an iteration has ended instead of polling for its residual.  Child processes, because the flag belongs to a
device's context."""
import json
import os
import subprocess
import sys

import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CHILD = """
import ctypes, json, sys, time
sys.path.insert(0, %r)
cuda = ctypes.CDLL("libcuda.so.1")
dev = ctypes.c_int()
assert cuda.cuInit(0) == 0 and cuda.cuDeviceGet(ctypes.byref(dev), 0) == 0
assert cuda.cuDevicePrimaryCtxSetFlags_v2(dev, int(sys.argv[1])) == 0
import torch
from paper_1201_5991_gb300 import meshgen
from paper_1201_5991_gb300.solver import BddcSolver
p = meshgen.elasticity3d(48, 4, seed=2)
s = BddcSolver(p, precision="mixed")
f = torch.tensor(p.f[:, 0], dtype=torch.float64, device="cuda")
u = s.solve(f, tol=1e-10)
w0, c0 = time.perf_counter(), time.thread_time()
for _ in range(20):
    v = s.solve(f, tol=1e-10)
print(json.dumps([(time.thread_time() - c0) / (time.perf_counter() - w0), bool(torch.equal(u, v)), float(v.norm())]))
"""


def _run(flags):
    out = subprocess.run([sys.executable, "-c", CHILD % ROOT, str(flags)], capture_output=True, text=True, timeout=300)
    assert out.returncode == 0, out.stderr[-2000:]
    return json.loads(out.stdout.strip().splitlines()[-1])


def test_blocking_and_yielding_waits():
    poll, block, give = _run(1), _run(4), _run(2)   # CU_CTX_SCHED_SPIN, _BLOCKING_SYNC, _YIELD
    print("host core used by the solving thread: polling %.2f, blocking %.2f, yielding %.2f" % (poll[0], block[0], give[0]))
    assert block[0] < 0.5
    assert poll[1] and block[1] and give[1] and poll[2] == block[2] == give[2]
