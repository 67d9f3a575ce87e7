"""Kernels that start while the one before them finishes read what it wrote: steps enqueued without a
synchronisation, with a sort (or an order-preserving repack) and the kinetic diagnostics after every step, equal
the same steps with the host waiting between the parts, bit for bit."""
import numpy as np
import pytest

import inputs as I
from paper_1608_04601_gb300 import xsections as X

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
@pytest.mark.parametrize("sort_every,spp", [(1, 400), (0, 67)])  # 67 steps a period: a repack after every step
def test_chained_equals_synchronised(prec, sort_every, spp):
    import __graft_entry__ as g
    g.build()
    from paper_1608_04601_gb300 import pic
    gas = X.he_like(eps_max_eV=300.0, de_eV=1e-2)
    d = I.discharge(n_cells=101, p_Pa=60.0, V_rf_V=200.0, n_e0=60001, n_i0=50002, n_init_m3=4e14, gamma_see=0.1,
                    steps_per_period=spp)
    got = []
    for chained in (True, False):
        sim = pic.Simulation(gas, d, seed=4, precision=prec, sort_every=sort_every if chained else 0)
        sim.set_diagnostics(period_steps=spp, phase_step=1, sample_every=1, eedf_bins=100, eedf_de_eV=0.5, fast_eV=20.0)
        if chained:
            sim.step(25)
        else:
            for _ in range(25):
                sim.step(1)
                sim.sync()
                if sort_every:
                    sim.sort()
                    sim.sync()
        got.append(([sim.get_state(0, sp) for sp in (0, 1)], sim.get_field(0)[1], sim.diagnostics(0), sim.moments(0)))
        sim.close()
    (sa, Ea, da, ma), (sb, Eb, db, mb) = got
    assert np.array_equal(Ea, Eb) and np.array_equal(ma["n_e"], mb["n_e"]) and ma["count"] == mb["count"]
    for sp in (0, 1):
        for k in ("c", "f", "vx", "vy", "vz"):
            assert np.array_equal(sa[sp][k], sb[sp][k]), (sp, k)
    for k in da:
        assert np.array_equal(da[k], db[k]), k
