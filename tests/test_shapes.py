"""Simulation.shape: whatever int() takes is an index, asked for once per lattice, and a closed context is
refused.  The library's calls are stood in for (no GPU needed)."""
import numpy as np
import pytest

from paper_1808_05168_gb300 import LatticeParams, Simulation, capi


def test_shapes_by_index_until_closed(monkeypatch):
    asked = []

    def shape(h, lattice):
        asked.append(int(lattice))
        if h is None:
            raise capi.LBError(capi.LB_ERR_BAD_PARAM, "lb_lattice_shape")
        return [(16, 8), (32, 4)][int(lattice)]

    monkeypatch.setattr(capi, "lb_create_batch", lambda params, flags: object())
    monkeypatch.setattr(capi, "lb_destroy", lambda h: None)
    monkeypatch.setattr(capi, "lb_lattice_shape", shape)
    sim = Simulation([LatticeParams(16, 8), LatticeParams(32, 4)])
    for one in (1, np.int64(1), np.array(1)):  # the last has no hash
        assert sim.shape(one) == (32, 4)
    i = np.array(0)
    assert sim.shape(i) == (16, 8)
    i += 1
    assert sim.shape(i) == (32, 4)
    assert asked == [1, 0]
    for _ in range(2):
        with pytest.raises(IndexError):
            sim.shape(2)
    assert asked == [1, 0, 2, 2]
    sim.close()
    with pytest.raises(capi.LBError):
        sim.shape(1)
