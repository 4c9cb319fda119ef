"""The first snapshot spectrum of a process made inside a caller's stream capture: the call is stream-ordered
and needs no set-up of its own, so it is captured like any other, and replays give the spectrum of what the
field holds then.  In a process of its own, since any earlier spectrum would not be the first."""
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

CHILD = """
import sys
import numpy as np, torch
from paper_1808_05168_gb300 import capi
call = getattr(capi, sys.argv[1])
Lx, Lz = 256, 64
rng = np.random.default_rng(5)
phi = torch.zeros((Lz, Lx), dtype=torch.float64, device="cuda")
out = torch.full_like(phi, float("nan"))
st = torch.cuda.Stream()
torch.cuda.synchronize()
g = torch.cuda.CUDAGraph()
with torch.cuda.graph(g, stream=st):
    call(phi.data_ptr(), Lx, Lz, out.data_ptr(), st.cuda_stream)
for _ in range(2):
    x = rng.standard_normal((Lz, Lx))
    phi.copy_(torch.from_numpy(x))
    torch.cuda.synchronize()
    with torch.cuda.stream(st):
        g.replay()
    torch.cuda.synchronize()
    want = np.abs(np.fft.fft2(x)) ** 2 / (Lx * Lz)
    np.testing.assert_allclose(out.cpu().numpy(), want, rtol=0, atol=1e-12 * want.max())
print("ok")
"""


@pytest.mark.parametrize("call", ["lb_power_spectrum", "lb_power_spectrum_noalloc"])
def test_first_call_inside_a_capture(call):
    r = subprocess.run([sys.executable, "-c", CHILD, call], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and r.stdout.strip().endswith("ok"), r.stdout + r.stderr
