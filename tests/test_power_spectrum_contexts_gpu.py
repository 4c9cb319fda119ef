"""The snapshot spectrum in a CUDA context of the program's own: the kernels' attributes and the fixed array of
the allocation-free entry belong to the context, so both entries work in the primary context, in two contexts
made one after the other on the same device, and in the primary one again.  In a process of its own."""
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

CHILD = """
import ctypes
import numpy as np
from paper_1808_05168_gb300 import capi
cu = ctypes.CDLL("libcuda.so.1")
u64 = ctypes.c_uint64
rng = np.random.default_rng(3)
fields = [rng.standard_normal((4, 8192)), rng.standard_normal((64, 64))]  # the first needs the attributes

def work():
    got = []
    for x in fields:
        a, b = u64(), u64()
        assert cu.cuMemAlloc_v2(ctypes.byref(a), ctypes.c_size_t(x.nbytes)) == 0
        assert cu.cuMemAlloc_v2(ctypes.byref(b), ctypes.c_size_t(x.nbytes)) == 0
        for call in (capi.lb_power_spectrum, capi.lb_power_spectrum_noalloc):
            assert cu.cuMemcpyHtoD_v2(a, x.ctypes.data_as(ctypes.c_void_p), ctypes.c_size_t(x.nbytes)) == 0
            call(a.value, x.shape[1], x.shape[0], b.value)
            assert cu.cuCtxSynchronize() == 0
            y = np.empty_like(x)
            assert cu.cuMemcpyDtoH_v2(y.ctypes.data_as(ctypes.c_void_p), b, ctypes.c_size_t(x.nbytes)) == 0
            got.append(y)
            want = np.abs(np.fft.fft2(x)) ** 2 / x.size
            np.testing.assert_allclose(y, want, rtol=0, atol=1e-12 * want.max())
        assert cu.cuMemFree_v2(a) == 0 and cu.cuMemFree_v2(b) == 0
    return got

dev, ctx = ctypes.c_int(), ctypes.c_void_p()
assert cu.cuInit(0) == 0 and cu.cuDeviceGet(ctypes.byref(dev), 0) == 0
assert cu.cuDevicePrimaryCtxRetain(ctypes.byref(ctx), dev) == 0 and cu.cuCtxSetCurrent(ctx) == 0
want = work()
for _ in range(2):
    own = ctypes.c_void_p()
    assert cu.cuCtxCreate_v2(ctypes.byref(own), 0, dev) == 0  # current from here on
    for a, b in zip(work(), want):
        assert np.array_equal(a, b)
    assert cu.cuCtxDestroy_v2(own) == 0
assert cu.cuCtxSetCurrent(ctx) == 0
for a, b in zip(work(), want):
    assert np.array_equal(a, b)
print("ok")
"""


def test_every_context_has_its_own():
    r = subprocess.run([sys.executable, "-c", CHILD], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and r.stdout.strip().endswith("ok"), r.stdout + r.stderr
