"""What follows the transforms of a sample (correlations, pressure profile, statistics) in one launch over a batch:
every lattice of a batch gives bit for bit what it gives alone, with numbers of tiles, rows and lattices that do
not fill the blocks, with and without correlations, launched directly and replayed."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

from paper_1808_05168_gb300 import LatticeParams, Simulation

SHAPES = [(32, 4), (64, 16), (32, 32), (128, 8), (32, 16), (32, 4), (64, 32), (32, 8), (64, 4)]


def _lattices():
    return [LatticeParams(Lx, Lz, kT=1e-5, G=0.4, grad_c0=0.01, seed=7, lattice_id=i) for i, (Lx, Lz) in enumerate(SHAPES)]


def _results(lattices, prec, corr, **kw):
    with Simulation(lattices, precision=prec, **kw) as sim:
        sim.set_tile(64, 4)
        sim.set_sampling(1, 2)
        if corr:
            sim.set_correlations(("c", "ux"), modes=(1, 3))
        sim.step(9)
        sim.synchronize()
        out = []
        for i in range(len(lattices)):
            r = [sim.profile(f, lattice=i)[0] for f in ("p", "c")] + [np.array(sim.mean_pressure(lattice=i)), np.array(sim.mass(lattice=i))]
            if corr:
                r += [sim.correlation(f, lattice=i)[0] for f in ("c", "ux")]
                r += [sim.mode_correlation("c", m, lattice=i)[0] for m in range(2)]
            out.append(r)
        return out


@pytest.mark.parametrize("corr", [False, True])
@pytest.mark.parametrize("prec", ["fp64", "dev32"])
@pytest.mark.parametrize("kw", [{}, {"graph": True}, {"persistent": True}])
def test_batch_equals_single_lattices(prec, corr, kw):
    lattices = _lattices()
    batch = _results(lattices, prec, corr, **kw)
    for p, got in zip(lattices, batch):
        (want,) = _results([p], prec, corr)
        for a, b in zip(got, want):
            assert np.array_equal(a, b)
