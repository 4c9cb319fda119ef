"""The default options' adjoint kernels at the edges of their variants: unit and general rates (the batch
takes the general form if any lattice does), lattices of two and three rows (every row or all but one
beside a wall), odd widths; against the oracle's dual numbers with the bounds of the adjoint's other tests."""
import numpy as np
import pytest

import oracle
from paper_1808_05168_gb300 import LatticeParams, Simulation

pytestmark = pytest.mark.gpu

UNIT = dict(lambda_s=1.0, lambda_e=1.0, lambda_q=1.0, lambda_eps=1.0)
GENERAL = dict(lambda_s=1.2, lambda_e=0.9, lambda_q=1.3, lambda_eps=0.8)


@pytest.mark.parametrize("prec,gtol", [("fp64", 1e-8), ("dev32", 3e-3)])
@pytest.mark.parametrize("rates", ["unit", "general", "mixed"])
def test_rates_and_short_lattices(rates, prec, gtol):
    kinds = {"unit": [UNIT] * 3, "general": [GENERAL] * 3, "mixed": [UNIT, GENERAL, UNIT]}[rates]
    shapes = [(33, 2), (16, 3), (7, 12)]
    ps = [LatticeParams(x, z, kT=1e-3, G=0.5, grad_c0=0.2 / z, lambda_d=0.8, seed=3 + i, lattice_id=i, **k)
          for i, ((x, z), k) in enumerate(zip(shapes, kinds))]
    with Simulation(ps, precision=prec) as sim:
        losses, grads = sim.pressure_shift_gradients(24, 7)
    for p, loss, g in zip(ps, losses, grads):
        want, o_g = oracle.pressure_shift_grad(p.Lx, p.Lz, 24, lambda_s=p.lambda_s, lambda_d=p.lambda_d,
                                               lambda_e=p.lambda_e, lambda_q=p.lambda_q, lambda_eps=p.lambda_eps, kT=p.kT,
                                               G=p.G, grad_c0=p.grad_c0, seed=p.seed, lattice_id=p.lattice_id)
        np.testing.assert_allclose(g, o_g, rtol=0, atol=gtol * np.max(np.abs(o_g)))
        assert abs(loss - want) <= (1e-10 if prec == "fp64" else 1e-4) * abs(want)


@pytest.mark.parametrize("prec", ["fp64", "dev32"])
def test_loss_does_not_depend_on_segments_or_mode(prec):
    """The pressures are summed step by step in one order: the loss alone (segments of 32 states), and with
    the gradient in segments of 1, 7 and 40 states, is the same number."""
    ps = [LatticeParams(34, 10, kT=1e-3, G=0.5, grad_c0=0.02, seed=2), LatticeParams(16, 6, kT=1e-4, G=0.3, seed=4, lattice_id=1)]
    with Simulation(ps, precision=prec) as sim:
        want, _ = sim.pressure_shift_gradients(40, 40, want_grad=False)
        for ckpt in (1, 7, 40):
            losses, _ = sim.pressure_shift_gradients(40, ckpt)
            assert np.array_equal(losses, want)
