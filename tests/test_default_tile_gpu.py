"""Default items of 64 columns (FP64 batches whose 128-column items would fill the SMs unevenly): the state,
bit for bit that of 128-column items, in every launch mode and with the method's options, and the gradient."""
import numpy as np
import pytest

pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1808_05168_gb300 import LatticeParams, Simulation


def _batch(Lx, Lz, n):
    return [LatticeParams(Lx, Lz, kT=1e-4, G=0.5, grad_c0=0.5 / Lz, seed=i + 3) for i in range(n)]


@pytest.mark.parametrize("Lx,Lz,n,prec,width", [
    (160, 96, 1, "fp64", 64), (161, 96, 1, "fp64", 64), (130, 64, 2, "fp64", 64), (160, 96, 4, "fp64", 64),
    (256, 128, 1, "fp64", 128), (64, 32, 1, "fp64", 128), (160, 96, 1, "dev32", 128),
    (66, 120, 3, "fp64", 128), (211, 105, 1, "fp64", 128), (259, 208, 1, "fp64", 64),
])
@pytest.mark.parametrize("kw", [{}, {"persistent": True}, {"graph": True}, {"astar": False, "noise_loc": True, "wall_fixed": True}])
def test_same_state_as_wide_items(Lx, Lz, n, prec, width, kw):
    got = []
    for tile in (None, (128, 2)):
        with Simulation(_batch(Lx, Lz, n), precision=prec, **kw) as sim:
            if tile:
                sim.set_tile(*tile)
            else:
                assert sim.tile()[0] == width
            sim.step(5)
            got.append([sim.populations(i) for i in range(n)])
    for a, b in zip(*got):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("Lx,Lz,n", [(160, 96, 1), (161, 96, 1), (130, 64, 2)])
def test_same_gradient_as_wide_items(Lx, Lz, n):
    got = []
    for tile in (None, (128, 1)):
        with Simulation(_batch(Lx, Lz, n), precision="fp64") as sim:
            if tile:
                sim.set_tile(*tile)
            got.append(sim.pressure_shift_gradients(30, 10))
    for a, b in zip(*got):
        assert np.array_equal(a, b)
