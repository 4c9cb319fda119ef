"""Statistics cleared between samples, with and without a wait for the device in between: the clears are done
when the call returns, so the sample that follows at once on the context's stream starts from zero."""
import numpy as np
import pytest

from paper_1808_05168_gb300 import LatticeParams, Simulation

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["fp64", "dev32"])
def test_reset_then_sample_at_once(prec):
    p = LatticeParams(1024, 512, kT=1e-5, G=0.5, grad_c0=0.0005, seed=4)

    def run(wait):
        with Simulation(p, precision=prec) as sim:
            sim.set_sampling(0, 1)  # the accumulators are made and cleared here
            sim.set_correlations(("c",), modes=(1,))
            out = []
            for _ in range(6):
                if wait:
                    torch.cuda.synchronize()
                sim.step(1)
                s, n = sim.structure_factor("c")
                c, nc = sim.correlation("c")
                assert n == 1 and nc == 1
                out += [s, c, sim.profile("p")[0]]
                sim.reset_statistics()
            return out

    for a, b in zip(run(False), run(True)):
        assert np.array_equal(a, b)
