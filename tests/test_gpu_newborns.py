"""Compaction of a round's newborns, bit for bit against the oracle: every electron is a candidate and about
half of the candidates ionize, so that most newborns move by a few places to where another lane's newborn
still stood (all must be read before any is written). Electrons and ions, chunks of 64, 128 and 256 slots,
newborns next to the electrodes among them (some are absorbed at birth)."""
import numpy as np
import pytest

import inputs as I
from oracle import oracle as O
from paper_1608_04601_gb300 import xsections as X

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,ppt", [("fp32", 2), ("fp32", 4), ("fp32", 8), ("fp64", 4), ("fp64", 8)])
def test_newborn_order(prec, ppt):
    import __graft_entry__ as g
    g.build()
    from paper_1608_04601_gb300 import pic
    eps = np.arange(20001) * 1e-2
    k = 1e-10 / np.sqrt(2 * I.E_CH * np.maximum(eps, 1e-9) / I.M_E)  # nu dt >> 1
    z = np.zeros_like(eps)
    gas = X.GasTables("forced", 4.0026 * I.AMU, (1e9,), 24.6, 1e-2, np.stack([k, z, np.where(eps > 24.6, k, 0.0)], 1),
                      np.stack([z, z], 1))
    cells, n = 64, 20011
    d = I.discharge(n_cells=cells)
    dt = np.float32 if prec == "fp32" else np.float64
    rng = np.random.default_rng(8 + ppt)
    e = I.energy_state(rng, n, cells, 30.0, 150.0, I.M_E, dt)
    sim = pic.Simulation(gas, d, precision=prec, load=False, ppt=ppt, capacity=[(100000, 100000)])
    ref = O.Oracle(gas, d, "f32" if prec == "fp32" else "f64", load=False)
    sim.set_state(0, 0, e)
    ref.set_state(0, e)
    E = I.random_field(rng, cells, 2e4, dt)
    for step in range(3):
        sim.set_field(0, E)
        ref.set_field(E)
        sim.sweep()
        ref.sweep()
        assert sim.counters(0) == ref.counters(), step
        assert step > 0 or sim.count(0, 1) > n // 4
        for sp in (0, 1):
            a, b = sim.get_state(0, sp), ref.get_state(sp)
            for key in ("c", "f", "vx", "vy", "vz"):
                assert np.array_equal(a[key], b[key]), (step, sp, key)
    sim.close()
