"""Per-step launches that overlap at their ends and take the step index from the host: against graphs and
persistent launches (which count on the device) bit for bit, with samples, state exchange and other work on
the stream between the steps, after a checkpoint, and captured by the caller into a graph of its own."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1808_05168_gb300 import LatticeParams, Simulation

P = [LatticeParams(64, 16, kT=1e-5, G=0.5, grad_c0=0.02, seed=4), LatticeParams(128, 8, kT=1e-5, G=0.3, seed=5, lattice_id=1)]


def _run(prec, splits, lattices=P, every=3, **kw):
    with Simulation(lattices, precision=prec, **kw) as sim:
        if every:
            sim.set_sampling(1, every)
        for n in splits:
            sim.step(n)
        sim.synchronize()
        out = [sim.populations(i) for i in range(len(lattices))]
        if every:
            out += [sim.structure_factor("c", lattice=i)[0] for i in range(len(lattices))]
        return out


@pytest.mark.parametrize("prec", ["fp64", "dev32"])
@pytest.mark.parametrize("splits", [(14,), (1, 1, 5, 7), (2, 12)])
def test_launch_modes_agree(prec, splits):
    want = _run(prec, (14,), graph=True)
    for kw in ({}, {"persistent": True}, {"persistent": True, "graph": True}, {"bulk": False}):
        for a, b in zip(_run(prec, splits, **kw), want):
            assert np.array_equal(a, b)


def test_state_exchange_and_other_work_between_steps():
    with Simulation(P[0], precision="dev32") as sim:
        st = torch.cuda.Stream()
        sim.set_stream(st)
        x = torch.zeros(1 << 22, device="cuda")
        torch.cuda.synchronize()
        for _ in range(6):
            sim.step(1)
            cols = sim.export_columns(0, 64)
            with torch.cuda.stream(st):
                x += 1  # other work of the stream
                cols = cols.clone()
            sim.import_columns(0, cols)
            st.synchronize() if _ == 3 else None
        got = sim.populations()
    assert np.array_equal(got, _run("dev32", (6,), lattices=[P[0]], every=0)[0])


def test_resumed_run_counts_on():
    want = _run("dev32", (11,), every=0)
    for kw in ({}, {"graph": True}, {"persistent": True}):
        with Simulation(P, precision="dev32") as sim:
            sim.step(5)
            buf = sim.save_checkpoint()
        with Simulation(P, precision="dev32", **kw) as sim:
            sim.step(2)
            sim.load_checkpoint(buf)
            sim.step(1)
            sim.step(5)
            for i in range(2):
                assert np.array_equal(sim.populations(i), want[i])


def test_captured_by_the_caller():
    """Two steps captured on the caller's stream and replayed: every replay goes on from the last."""
    with Simulation(P[0], precision="dev32") as sim:
        st = torch.cuda.Stream()
        sim.set_stream(st)
        sim.step(2)
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=st):
            sim.step(2)
        with torch.cuda.stream(st):
            for _ in range(3):
                g.replay()
        torch.cuda.synchronize()
        got = sim.populations()
    assert np.array_equal(got, _run("dev32", (8,), lattices=[P[0]], every=0)[0])


@pytest.mark.parametrize("kw", [{}, {"persistent": True}])
def test_steps_after_replays_of_the_callers_graph(kw):
    """Steps called directly between and after such replays go on from what the replays have run."""
    with Simulation(P[0], precision="dev32", **kw) as sim:
        st = torch.cuda.Stream()
        sim.set_stream(st)
        sim.step(2)
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=st):
            sim.step(2)
        with torch.cuda.stream(st):
            for _ in range(3):
                g.replay()
        sim.step(2)
        with torch.cuda.stream(st):
            g.replay()
        sim.step(3)
        torch.cuda.synchronize()
        got = sim.populations()
    assert np.array_equal(got, _run("dev32", (15,), lattices=[P[0]], every=0)[0])
