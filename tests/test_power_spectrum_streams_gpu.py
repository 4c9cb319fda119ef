"""Snapshot spectra on several streams in turn: the right results, and calls that take no longer than on one
stream (where the scratch of other streams in flight made each wait in the allocator for 100 us)."""
import time

import numpy as np
import pytest

from paper_1808_05168_gb300 import capi

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _states(Lx, Lz, n):
    g = torch.Generator(device="cuda")
    g.manual_seed(Lx + Lz)
    out = []
    for _ in range(n):
        x = torch.randn((Lz, Lx), generator=g, dtype=torch.float64, device="cuda")
        out.append((x, torch.full_like(x, float("nan")), torch.cuda.Stream()))
    torch.cuda.synchronize()
    return out


def _turns(states, n):
    for i in range(n):
        x, out, s = states[i % len(states)]
        capi.lb_power_spectrum(x.data_ptr(), x.shape[1], x.shape[0], out.data_ptr(), s.cuda_stream)


@pytest.mark.parametrize("Lx,Lz", [(2, 2), (64, 256), (512, 256), (2048, 1024)])
def test_streams_in_turn(Lx, Lz):
    states = _states(Lx, Lz, 5)
    _turns(states, 60)
    torch.cuda.synchronize()
    for x, out, _ in states:
        x = x.cpu().numpy()
        want = np.abs(np.fft.fft2(x)) ** 2 / x.size
        np.testing.assert_allclose(out.cpu().numpy(), want, rtol=0, atol=1e-12 * want.max())


def test_calls_do_not_wait_for_other_streams():
    def per_call(states):
        best = float("inf")
        for _ in range(5):
            torch.cuda.synchronize()
            t = time.perf_counter()
            _turns(states, 300)
            torch.cuda.synchronize()
            best = min(best, (time.perf_counter() - t) / 300)
        return best

    states = _states(64, 256, 3)
    # three streams overlap: less than half of one stream's time per call (8 of 17 us; 108 in the allocator)
    assert per_call(states) < 1.5 * per_call(states[:1])
