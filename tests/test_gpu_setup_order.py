"""Set-up work is ordered with the context's stream.

A context's tables, counts and cleared deposits are written on the stream that its kernels run on.
Copies on another stream would race with the queued clears of large buffers: the voltage table of a
discharge could be cleared after it was written (the driven electrode then stays at 0 V), and the
deposits of the last discharges of a batch could be cleared while the warm load adds to them.
"""
import math

import numpy as np
import pytest

from paper_1608_04601_gb300 import xsections as X
from paper_1608_04601_gb300.workloads import Discharge

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    import __graft_entry__ as g
    g.build()
    from paper_1608_04601_gb300 import pic
    return pic


def _batch():
    # uneven stores with roomy capacities: hundreds of MB of scratch are cleared at create
    ns = [int(1e5 * 40 ** (i / 11)) for i in range(12)]
    return [Discharge("order", "ar", 0.025, 10.0, 300.0 + i, 512, 2000, n, n, 4e15, discharge_id=i)
            for i, n in enumerate(ns)]


def test_voltage_tables_survive_large_scratch(P):
    gas, ds = X.ar_like(eps_max_eV=200.0, de_eV=1e-2), _batch()
    sim = P.Simulation(gas, ds, seed=3, sort_every=16, capacity=[d.capacity(3.0) for d in ds])
    sim.step(3)
    for i, d in enumerate(ds):
        v = d.V_rf_V * math.sin(2 * math.pi * d.f_rf_Hz * 3 * d.dt_s)
        assert abs(sim.get_field(i)[2][0] - v) <= 1e-9 * abs(v), i
    sim.close()


def test_warm_load_of_a_batch_equals_single_loads(P):
    gas, ds = X.ar_like(eps_max_eV=200.0, de_eV=1e-2), _batch()
    z = np.linspace(0.0, 1.0, 65)
    prof = np.stack([4e15 * np.sin(np.pi * z) + 1e14, 4e15 * np.sin(np.pi * z) + 2e14, np.full(65, 3.0)])
    sim = P.Simulation(gas, ds, seed=3, load=False)
    sim.load_profiles(np.stack([prof] * len(ds)))
    fields = [sim.get_field(i)[1] for i in range(len(ds))]
    sim.close()
    for i, d in enumerate(ds):
        one = P.Simulation(gas, d, seed=3, load=False)
        one.load_profiles(prof)
        assert np.array_equal(one.get_field(0)[1], fields[i]), i
        one.close()
