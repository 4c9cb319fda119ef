"""The double-precision inverse transform in integers of one scale, where it scales differently or steps
aside: a species of zero, of tiny and of very tiny density beside a normal one, populations of mixed
magnitudes, infinities and NaN; against the oracle."""
import numpy as np
import pytest

import oracle
from paper_1808_05168_gb300 import LatticeParams, Simulation

pytestmark = pytest.mark.gpu

W = np.array([4 / 9] + [1 / 9] * 4 + [1 / 36] * 4)


def _state(Lx, Lz, scale):
    rng = np.random.default_rng(3)
    f = W[None, :, None, None] * (0.5 + 0.05 * rng.standard_normal((2, 9, Lz, Lx)))
    f[1] *= scale
    return f


def _run(scale, bulk):
    # no coupling, gradient or noise: species B enters its own update linearly
    f = _state(32, 6, scale)
    with Simulation(LatticeParams(32, 6, lambda_s=1.2, lambda_d=0.9), bulk=bulk) as sim:
        sim.set_populations(f)
        sim.step(3)
        return f, sim.populations()


@pytest.mark.parametrize("bulk", [True, False])
@pytest.mark.parametrize("scale", [1.0, 2.0 ** -40])
def test_species_of_unequal_magnitude(scale, bulk):
    f, got = _run(scale, bulk)
    o = oracle.OracleLattice(32, 6, lambda_s=1.2, lambda_d=0.9, kT=0.0, G=0.0, grad_c0=0.0)
    o.set_populations(f)
    o.step(3)
    want = o.populations()
    for s in range(2):
        # the parity bar of FP64 populations, against the species' own magnitude
        assert np.max(np.abs(got[s] - want[s])) <= 1e-12 * np.max(np.abs(want[s]))


@pytest.mark.parametrize("bulk", [True, False])
def test_species_of_vanishing_density(bulk):
    """Beside a normal species A (the oracle divides by 1 - c and has no value there): B scales with its
    density, through the integers and, below their range, in double; A does not see it; zero stays zero."""
    _, near = _run(2.0 ** -40, bulk)
    _, small = _run(2.0 ** -300, bulk)
    _, tiny = _run(2.0 ** -960, bulk)
    _, none = _run(0.0, bulk)
    # a density of 2^-40 changes the velocity by 2^-40 of it, below the parity bar of 1e-12
    assert np.max(np.abs(small[1] * 2.0 ** 260 - near[1])) <= 1e-12 * np.max(near[1])
    assert np.max(np.abs(tiny[1] * 2.0 ** 660 - small[1])) <= 1e-12 * np.max(small[1])
    assert np.array_equal(tiny[0], small[0]) and np.array_equal(none[0], small[0])
    assert not none[1].any()


@pytest.mark.parametrize("bad", [np.nan, np.inf, 1e308])
def test_values_beyond_the_scale(bad):
    p = LatticeParams(32, 6, lambda_s=1.2, lambda_d=0.9)
    f = _state(32, 6, 1.0)
    f[0, 5, 3, 7] = bad
    with Simulation(p) as sim:
        sim.set_populations(f)
        sim.step(1)
        got = sim.populations()
    x, z = 8, 4  # link 5 moves one column and one row
    touched = np.zeros((6, 32), bool)
    touched[z - 1:z + 2, x - 1:x + 2] = True
    assert np.isfinite(got[:, :, ~touched]).all()  # only the site it arrives at (and, by the force, around it)
    there = got[0, :, z, x]
    if bad == 1e308:  # one population beyond the scale: the double arithmetic, no wrapped integer
        assert (~np.isfinite(there)).any() or np.max(np.abs(there)) > 1e300
    else:
        assert not np.isfinite(there).all()
