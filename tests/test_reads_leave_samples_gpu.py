"""Reading results changes no buffer that a sample step works with, so a sampling step that the caller has
captured and replays on another stream is not disturbed by a read meanwhile: of the context's buffers (all from
the test's allocator), those that the reads change and those that a sample step changes have none in common."""

import pytest

from paper_1808_05168_gb300 import LatticeParams, Simulation, capi

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["fp64", "dev32"])
def test_reads_and_samples_share_no_buffer(prec):
    held = {}

    def alloc(nbytes, user):
        t = torch.zeros((int(nbytes) + 511) // 256 * 256, dtype=torch.uint8, device="cuda")
        at = (-t.data_ptr()) % 256
        held[t.data_ptr() + at] = t
        return t.data_ptr() + at

    def free(ptr, user):
        held.pop(ptr)

    def changed(work):
        torch.cuda.synchronize()
        before = {p: t.clone() for p, t in held.items()}
        work()
        torch.cuda.synchronize()
        return {p for p, t in before.items() if not torch.equal(t, held[p])}

    ps = [LatticeParams(16, 8, kT=1e-5, G=0.5, grad_c0=0.03, seed=3, lattice_id=i) for i in range(2)]
    cb = capi.LB_ALLOC_FN(alloc), capi.LB_FREE_FN(free)
    with Simulation(ps, precision=prec, allocator=cb) as sim:
        sim.set_sampling(0, 1)
        sim.set_correlations(("c",), modes=(1,))
        sim.step(3)
        sim.synchronize()

        def reads():
            for i in range(2):
                sim.structure_factor("c", lattice=i)
                sim.structure_factor("rho", lattice=i, qz0_only=True)
                sim.profile("p", lattice=i)
                sim.correlation("c", lattice=i)
                sim.mode_correlation("c", 0, lattice=i)
                sim.mean_pressure(i)

        def sample():
            sim.step(1)
            sim.synchronize()

        by_reads, by_sample = changed(reads), changed(sample)
        assert by_sample and not by_reads & by_sample
    assert not held
