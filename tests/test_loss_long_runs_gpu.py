"""Runs so long that the steps' pressures reach the host in several pieces (65536 values, so 32768 steps of two
lattices): each lattice's loss is that of a context that holds it alone, whose pieces end elsewhere, bit for
bit; and the last piece of one step."""
import numpy as np
import pytest

from paper_1808_05168_gb300 import LatticeParams, Simulation

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["fp64", "dev32"])
@pytest.mark.parametrize("steps", [32769, 40000])
def test_losses_of_long_runs(prec, steps):
    ps = [LatticeParams(4, 4, kT=1e-5, G=0.5, grad_c0=0.05, seed=3 + i, lattice_id=i) for i in range(2)]
    with Simulation(ps, precision=prec) as sim:
        both = sim.pressure_shift_gradients(steps, steps, want_grad=False)[0]
    assert np.all(np.isfinite(both)) and both[0] != both[1]
    for p, want in zip(ps, both):
        with Simulation(p, precision=prec) as sim:
            assert sim.pressure_shift_gradient(steps, steps, want_grad=False)[0] == want
