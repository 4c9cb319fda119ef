"""The persistent launch with a block per item (each block keeps its item) against per-step launches, bit for
bit: one-row items, a last chunk that is shorter, a batch of equal lattices, and lattices of one and of two
chunk lengths (the second goes by tickets)."""
import numpy as np
import pytest

from paper_1808_05168_gb300 import LatticeParams, Simulation

pytestmark = pytest.mark.gpu


def _run(shapes, prec, tile, persistent, bulk=True):
    ps = [LatticeParams(x, z, kT=1e-5, G=0.5, grad_c0=0.3 / z, seed=4, lattice_id=i) for i, (x, z) in enumerate(shapes)]
    with Simulation(ps, precision=prec, persistent=persistent, bulk=bulk) as sim:
        sim.set_tile(*tile)
        sim.step(7)
        sim.step(6)
        return [sim.populations(i) for i in range(len(ps))]


@pytest.mark.parametrize("prec", ["fp64", "dev32"])
@pytest.mark.parametrize("shapes,tile,bulk", [([(64, 32)], (128, 1), True), ([(300, 17)], (64, 3), True), ([(2, 2)], (32, 1), True),
                                              ([(96, 8)] * 3, (32, 2), True), ([(96, 8), (64, 16)], (32, 8), True),
                                              ([(96, 8), (64, 16)], (32, 16), True), ([(65, 9)], (32, 2), False)])
def test_equals_per_step_launches(shapes, tile, prec, bulk):
    want = _run(shapes, prec, tile, False, bulk)
    got = _run(shapes, prec, tile, True, bulk)
    for w, g in zip(want, got):
        assert np.array_equal(w, g)
