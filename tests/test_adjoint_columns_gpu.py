"""The gradient's noiseless run on two columns: lattices of one, two and odd numbers of columns, and a
lattice without noise inside a noisy batch (whose two runs are the same run)."""
import numpy as np
import pytest

import oracle
from paper_1808_05168_gb300 import LatticeParams, Simulation

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("Lx", [1, 2, 5, 33])
def test_any_width_matches_oracle(Lx):
    p = LatticeParams(Lx, 6, kT=1e-3, G=0.5, grad_c0=0.05, lambda_s=1.2, lambda_d=0.9, lambda_e=1.0, seed=5)
    with Simulation(p) as sim:
        loss, g = sim.pressure_shift_gradient(20, 6)
    o_loss, o_g = oracle.pressure_shift_grad(p.Lx, p.Lz, 20, lambda_s=p.lambda_s, lambda_d=p.lambda_d,
                                             lambda_e=p.lambda_e, kT=p.kT, G=p.G, grad_c0=p.grad_c0, seed=p.seed)
    # the bounds of the adjoint's other comparisons with the oracle (FP64 sums of 20 steps)
    assert abs(loss - o_loss) <= 1e-10 * abs(o_loss)
    np.testing.assert_allclose(g, o_g, rtol=0, atol=1e-8 * np.max(np.abs(o_g)))


@pytest.mark.parametrize("prec", ["fp64", "dev32"])
def test_lattice_without_noise_in_a_noisy_batch(prec):
    ps = [LatticeParams(16, 8, kT=k, G=0.5, grad_c0=0.03, seed=3, lattice_id=i) for i, k in enumerate((1e-3, 0.0))]
    with Simulation(ps, precision=prec) as sim:
        losses, grads = sim.pressure_shift_gradients(12, 5)
    assert losses[0] != 0.0 and np.all(grads[0] != 0.0)
    assert losses[1] == 0.0 and np.all(grads[1] == 0.0)
