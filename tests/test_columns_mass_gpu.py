"""Column blocks of the stored state and the masses at the sizes where their kernels change hands: column
counts around the width that a block takes one row of, and lattices of an odd number of sites, of one
block and of several."""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1808_05168_gb300 import LatticeParams, Simulation


def _sim(Lx, Lz, prec):
    return Simulation(LatticeParams(Lx, Lz, grad_c0=0.3 / Lz), precision=prec)


@pytest.mark.parametrize("prec", ["fp64", "dev32"])
@pytest.mark.parametrize("Lx", [127, 128, 1024, 1025])
def test_columns_round_trip(prec, Lx):
    Lz = 3
    dt = torch.float64 if prec == "fp64" else torch.float32
    g = torch.Generator().manual_seed(Lx)
    want = torch.rand((18, Lz, Lx), generator=g, dtype=dt)
    with _sim(Lx, Lz, prec) as sim:
        sim.import_columns(0, want.cuda())
        for first, n in ((0, Lx), (1, Lx - 1), (Lx - 2, 2), (0, 1), (max(0, Lx - 128), 127)):
            got = sim.export_columns(first, n)
            sim.synchronize()
            assert torch.equal(got.cpu(), want[:, :, first:first + n])
        if prec == "fp64":  # no background: the absolute populations are the stored values
            assert np.array_equal(sim.populations().reshape(18, Lz, Lx), want.numpy())
        # a narrow block overwritten in the middle leaves the rest alone
        cols = torch.rand((18, Lz, 5), generator=g, dtype=dt)
        sim.import_columns(60, cols.cuda())
        want[:, :, 60:65] = cols
        got = sim.export_columns(0, Lx)
        sim.synchronize()
        assert torch.equal(got.cpu(), want)


@pytest.mark.parametrize("prec", ["fp64", "dev32"])
@pytest.mark.parametrize("Lx, Lz", [(1, 2), (3, 5), (61, 37), (333, 119), (1024, 130)])
def test_mass(prec, Lx, Lz):
    """Against the exact sum of the populations; every sum runs over at most about a hundred terms in a
    row (per thread, per block, over the blocks): 100 eps relative."""
    dt = torch.float64 if prec == "fp64" else torch.float32
    x = torch.rand((18, Lz, Lx), generator=torch.Generator().manual_seed(Lx + Lz), dtype=dt) * 0.01
    with _sim(Lx, Lz, prec) as sim:
        sim.import_columns(0, x.cuda())
        f = sim.populations().reshape(2, -1)
        for _ in range(2):  # the block counter is left as it was found
            m = sim.mass()
            for s in range(2):
                assert abs(m[s] - math.fsum(f[s])) <= 100 * 2.3e-16 * m[s]
