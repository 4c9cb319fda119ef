"""A gradient call on a context with the caller's allocator waits for its own work, not for the device: it
returns while another (non-blocking) stream of the program is still busy, with the same results."""
import numpy as np
import pytest

from paper_1808_05168_gb300 import LatticeParams, Simulation

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("want_grad", [True, False])
@pytest.mark.parametrize("prec", ["fp64", "dev32"])
def test_returns_while_another_stream_works(prec, want_grad):
    with Simulation(LatticeParams(32, 8, kT=1e-4, G=0.5, grad_c0=0.03, seed=3), precision=prec, allocator="torch") as sim:
        for _ in range(2):  # modules loaded, the allocator's blocks cached
            want = sim.pressure_shift_gradient(6, 3, want_grad)
        other, done = torch.cuda.Stream(), torch.cuda.Event()
        torch.cuda.synchronize()
        with torch.cuda.stream(other):
            torch.cuda._sleep(3_000_000_000)  # clocks: more than a second; the call takes milliseconds
            done.record()
        got = sim.pressure_shift_gradient(6, 3, want_grad)
        busy = not done.query()
        torch.cuda.synchronize()
    assert busy
    assert got[0] == want[0] and (not want_grad or np.array_equal(got[1], want[1]))
