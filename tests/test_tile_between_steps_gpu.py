"""A new tile while steps are in flight: they finish on the items they were launched with (set_tile waits for
them), and the states are those of an undisturbed run, bit for bit, with one launch per step and persistent."""
import numpy as np
import pytest

from paper_1808_05168_gb300 import LatticeParams, Simulation

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("persistent", [False, True])
@pytest.mark.parametrize("prec", ["fp64", "dev32"])
def test_tiles_changed_between_steps(prec, persistent):
    p = LatticeParams(300, 64, kT=1e-5, G=0.5, grad_c0=0.005, seed=4)
    with Simulation(p, precision=prec) as sim:
        sim.step(1200)
        want = sim.populations()
    with Simulation(p, precision=prec, persistent=persistent) as sim:
        for tile in ((128, 64), (32, 1), (256, 3), (64, 7)):
            sim.set_tile(*tile)
            sim.step(300)
        assert np.array_equal(sim.populations(), want)
