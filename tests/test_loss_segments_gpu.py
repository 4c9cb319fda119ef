"""The loss alone runs in segments of states that go up a ring and down again; the gradient's forward run goes
from checkpoint to checkpoint.  Both sum the same pressures in the same order, so the losses are equal bit for
bit: segments of 32 states that end early, on the last state and one after it, on bulk and per-thread staging,
and states so large that a segment holds one of them or three."""
import numpy as np
import pytest

from paper_1808_05168_gb300 import LatticeParams, Simulation

pytestmark = pytest.mark.gpu


def _losses(shapes, prec, steps, ckpt):
    ps = [LatticeParams(x, z, kT=1e-4, G=0.5, grad_c0=0.3 / z, seed=3, lattice_id=i) for i, (x, z) in enumerate(shapes)]
    with Simulation(ps, precision=prec) as sim:
        alone = sim.pressure_shift_gradients(steps, ckpt, want_grad=False)[0]
        return np.array(alone), np.array(sim.pressure_shift_gradients(steps, ckpt)[0])


@pytest.mark.parametrize("prec", ["fp64", "dev32"])
@pytest.mark.parametrize("steps", [1, 2, 32, 33, 64, 65, 100])
@pytest.mark.parametrize("shapes", [[(32, 8)], [(17, 5), (24, 6)]])
def test_segments(shapes, steps, prec):
    alone, with_gradient = _losses(shapes, prec, steps, min(steps, 9))
    assert np.array_equal(alone, with_gradient) and np.all(np.isfinite(alone))


@pytest.mark.parametrize("prec,Lx,Lz,steps", [("fp64", 2048, 2048, 5), ("dev32", 2048, 4096, 4), ("fp64", 1024, 2048, 8)])
def test_large_states(prec, Lx, Lz, steps):
    alone, with_gradient = _losses([(Lx, Lz)], prec, steps, steps)
    assert np.array_equal(alone, with_gradient) and np.all(np.isfinite(alone))
