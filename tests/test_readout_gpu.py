"""Results read through one launch and one copy: spectra, profiles, correlations and pressures equal what the
checkpoint's raw sums give, bit for bit, for a first lattice and a later one, a spectrum short and longer than
the single copy takes, its q_z = 0 row, and correlations that do and do not fit the buffer."""
import numpy as np
import pytest

from paper_1808_05168_gb300 import LatticeParams, Simulation, capi

pytestmark = pytest.mark.gpu


def _sums(sim, shapes, modes):
    """The accumulators in the order of a checkpoint (the end of it): spectra, profiles, correlations."""
    buf = sim.save_checkpoint()
    sites, rows = sum(x * z for x, z in shapes), sum(z for _, z in shapes)
    sizes = [4 * sites, 4 * sites, 5 * rows, 5 * rows, sum(4 * z * z for _, z in shapes),
             sum(8 * modes * z * z for _, z in shapes)]
    raw = buf[len(buf) - 8 * sum(sizes):].view(np.float64)
    return np.split(raw, np.cumsum(sizes)[:-1])


@pytest.mark.parametrize("prec", ["fp64", "dev32"])
@pytest.mark.parametrize("shapes", [[(16, 4), (32, 8)], [(2, 2)], [(256, 256)], [(4, 128)]])
def test_results_equal_the_raw_sums(shapes, prec):
    ps = [LatticeParams(x, z, kT=1e-5, G=0.5, grad_c0=0.3 / z, seed=3, lattice_id=i) for i, (x, z) in enumerate(shapes)]
    with Simulation(ps, precision=prec) as sim:
        sim.set_sampling(0, 2)
        sim.set_correlations(("c", "ux"), modes=(1,))
        sim.step(5)
        s, k, ps_, pk, R, C = _sums(sim, shapes, 1)
        so = ro = co = 0
        rows = sum(z for _, z in shapes)
        for i, (Lx, Lz) in enumerate(shapes):
            n = Lx * Lz
            for f, name in enumerate(("rho", "c", "ux", "uz")):
                acc = (s[4 * so + f * n:4 * so + (f + 1) * n] - k[4 * so + f * n:4 * so + (f + 1) * n]).reshape(Lz, Lx) * (1.0 / 3)
                want = acc.copy()
                for q in range(Lx // 2 + 1, Lx):
                    want[:, q] = acc[(-np.arange(Lz)) % Lz, Lx - q]
                got, cnt = sim.structure_factor(name, lattice=i)
                assert cnt == 3 and np.array_equal(got, want)
                assert np.array_equal(sim.structure_factor(name, lattice=i, qz0_only=True)[0], want[0])
            p = (ps_[2 * rows + ro:2 * rows + ro + Lz] + pk[2 * rows + ro:2 * rows + ro + Lz]) * (1.0 / 3)
            assert np.array_equal(sim.profile("ux", lattice=i)[0], p)
            assert np.array_equal(sim.correlation("c", lattice=i)[0].ravel(), R[co + Lz * Lz:co + 2 * Lz * Lz] * (1.0 / 3))
            c = C[2 * co + 2 * Lz * Lz:2 * co + 4 * Lz * Lz] * (1.0 / 3)
            assert np.array_equal(sim.mode_correlation("c", 0, lattice=i)[0].ravel(), c[0::2] + 1j * c[1::2])
            last, avg = sim.mean_pressure(i)
            assert abs(avg - sim.profile("p", lattice=i)[0].mean()) <= 1e-7 * abs(avg) and np.isfinite(last)
            so, ro, co = so + n, ro + Lz, co + 4 * Lz * Lz
    with pytest.raises(capi.LBError):
        with Simulation(ps, precision=prec) as sim:
            sim.shape(len(ps))
