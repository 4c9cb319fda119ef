"""The FP64 normals' tables belong to the CUDA context that uses them: a program that works in the primary
context, then in contexts of its own made one after the other on the same device, gets the same normals and
the same steps in each.  In a process of its own, which leaves the test process's context alone."""
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

CHILD = """
import ctypes
import numpy as np
from paper_1808_05168_gb300 import LatticeParams, Simulation, capi
words = np.random.default_rng(3).integers(0, 1 << 32, 4096, dtype=np.uint64).astype(np.uint32)

def work():
    n = capi.lb_debug_box_muller(capi.LB_PREC_FP64, words)
    with Simulation(LatticeParams(32, 8, kT=1e-5, G=0.5, grad_c0=0.02, seed=4), precision="fp64") as sim:
        sim.step(3)
        return n, sim.populations()

want = work()
assert abs(float(np.std(want[0])) - 1.0) < 0.1
cu = ctypes.CDLL("libcuda.so.1")
dev = ctypes.c_int()
assert cu.cuInit(0) == 0 and cu.cuDeviceGet(ctypes.byref(dev), 0) == 0
for _ in range(2):
    ctx = ctypes.c_void_p()
    assert cu.cuCtxCreate_v2(ctypes.byref(ctx), 0, dev) == 0  # current from here on
    for a, b in zip(work(), want):
        assert np.array_equal(a, b)
    assert cu.cuCtxDestroy_v2(ctx) == 0
for a, b in zip(work(), want):  # the primary context again
    assert np.array_equal(a, b)
print("ok")
"""


def test_every_context_has_its_own_tables():
    r = subprocess.run([sys.executable, "-c", CHILD], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and r.stdout.strip().endswith("ok"), r.stdout + r.stderr
