"""Persistent launches of two contexts at the same time, from two threads on two streams: grids whose blocks
keep their items (one row each, up to a block per SM), grids that take tickets, and one of each, in both
precisions; the states are those of one launch per step, bit for bit."""
import threading

import numpy as np
import pytest

from paper_1808_05168_gb300 import LatticeParams, Simulation

pytestmark = pytest.mark.gpu

OWNED = ((64, 152), 1, (128, 1))    # 152 items
BATCH = ((128, 32), 4, (128, 1))    # 128 items
TICKETS = ((512, 160), 1, (128, 1))  # 640 items


def _run(what, prec, seed, persistent, gate=None):
    (x, z), n, tile = what
    ps = [LatticeParams(x, z, kT=1e-5, G=0.5, grad_c0=0.3 / z, seed=seed, lattice_id=i) for i in range(n)]
    with Simulation(ps, precision=prec, persistent=persistent) as sim:
        sim.set_tile(*tile)
        sim.step(2)
        sim.synchronize()
        if gate:
            gate.wait()
        for i in range(40):
            sim.step(25)
            if i % 8 == 7:
                sim.synchronize()
        sim.synchronize()
        return [sim.populations(i) for i in range(n)]


@pytest.mark.parametrize("one,two", [((OWNED, "fp64"), (OWNED, "fp64")), ((OWNED, "fp64"), (BATCH, "dev32")),
                                     ((BATCH, "dev32"), (BATCH, "dev32")), ((TICKETS, "dev32"), (OWNED, "fp64")),
                                     ((TICKETS, "fp64"), (TICKETS, "dev32"))])
def test_two_contexts_at_once(one, two):
    jobs, gate, got, failed = [one, two], threading.Barrier(2, timeout=120), [None, None], []

    def work(i):
        try:
            got[i] = _run(*jobs[i], 7 + i, True, gate)
        except Exception as e:  # noqa: BLE001
            failed.append(e)

    threads = [threading.Thread(target=work, args=(i,)) for i in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failed, failed
    for i in range(2):
        for a, b in zip(got[i], _run(*jobs[i], 7 + i, False)):
            assert np.array_equal(a, b)
