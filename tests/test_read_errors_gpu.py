"""A read that finds the device's error flag set returns LB_ERR_TIMEOUT and leaves the caller's buffer as it
was, for results that are copied with the flag and for long ones; the next read is served.  The flag is set
from the host, through the test's allocator (the only four-byte buffer of a context)."""
import numpy as np
import pytest

from paper_1808_05168_gb300 import LatticeParams, Simulation, capi

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("Lx,Lz", [(16, 8), (256, 256)])
def test_a_flagged_read_leaves_the_buffer_alone(Lx, Lz):
    held, sizes = {}, {}

    def alloc(nbytes, user):
        t = torch.zeros(int(nbytes) + 256, dtype=torch.uint8, device="cuda")
        p = t.data_ptr() + (-t.data_ptr()) % 256
        held[p], sizes[p] = t, int(nbytes)
        return p

    def free(ptr, user):
        del held[ptr]

    cb = capi.LB_ALLOC_FN(alloc), capi.LB_FREE_FN(free)
    with Simulation(LatticeParams(Lx, Lz, kT=1e-5, G=0.5, seed=3), precision="dev32", allocator=cb) as sim:
        sim.set_sampling(0, 1)
        sim.step(2)
        want = sim.structure_factor("c")[0]
        flags = [p for p in held if sizes[p] == 4]
        assert len(flags) == 1
        at = flags[0] - held[flags[0]].data_ptr()
        held[flags[0]][at] = 1
        torch.cuda.synchronize()
        out = np.full((Lz, Lx), -1.0)
        with pytest.raises(capi.LBError) as e:
            capi.lb_structure_factor(sim.h, 0, capi.LB_FIELD_C, capi.LB_SF_QXQZ, out)
        assert e.value.code == capi.LB_ERR_TIMEOUT and np.all(out == -1.0)
        capi.lb_structure_factor(sim.h, 0, capi.LB_FIELD_C, capi.LB_SF_QXQZ, out)
        assert np.array_equal(out, want)
