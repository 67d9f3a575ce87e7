"""The sweep at the edges of its dispatch, bit for bit against the oracle.

Cell counts around the histogram window (64 cells) and where a CTA holds one species' histograms at a
time (above about 2900 cells), stores with and without a window (16 chunks per CTA), chunks of 64, 128
and 256 slots, stores that end in the middle of a row, electrons of every energy (the part above 32 eV
of the energy moment takes another array where it fits, or goes to the global sums: 2047 cells). Each step starts on both sides from the same state and field.
"""
import numpy as np
import pytest

import inputs as I
from oracle import oracle as O
from paper_1608_04601_gb300 import xsections as X

pytestmark = pytest.mark.gpu

# precision, cells, particles per thread, electrons, ions, steps before and after a sort
CASES = [("fp32", 1, 4, 1000, 777, 2), ("fp32", 63, 2, 3001, 129, 3), ("fp32", 64, 4, 420001, 380003, 2),
         ("fp32", 65, 8, 5000, 4999, 3), ("fp32", 1700, 4, 480001, 470003, 2), ("fp32", 2047, 4, 480001, 470003, 2),
         ("fp32", 2900, 4, 40001, 30011, 2), ("fp32", 4096, 4, 340007, 330001, 2),
         ("fp32", 4096, 8, 9000, 8001, 2), ("fp64", 64, 4, 30001, 20003, 2), ("fp64", 1500, 2, 180001, 170003, 2),
         ("fp64", 4096, 4, 20001, 20002, 2), ("fp64", 4096, 8, 9001, 9002, 2)]


@pytest.fixture(scope="module")
def P():
    import __graft_entry__ as g
    g.build()
    from paper_1608_04601_gb300 import pic
    return pic


@pytest.mark.parametrize("case", CASES, ids=["-".join(map(str, c)) for c in CASES])
def test_sweep_bit_exact(P, case):
    prec, cells, ppt, ne, ni, steps = case
    rng = np.random.default_rng(cells + ppt)
    dt = np.float32 if prec == "fp32" else np.float64
    gas = X.he_like(eps_max_eV=200.0, de_eV=1e-2)
    d = I.discharge(n_cells=cells, p_Pa=200.0, gamma_see=0.2, n_e0=1, n_i0=1, V_rf_V=100.0)
    cap = [(2 * ne + 8192, 2 * ni + ne + 8192)]
    sim = P.Simulation(gas, d, precision=prec, load=False, ppt=ppt, capacity=cap)
    ref = O.Oracle(gas, d, "f32" if prec == "fp32" else "f64", load=False)
    st = [I.mixed_state(rng, n, cells, sp, dt, d.gap_m, d.dt_s) for sp, n in ((0, ne), (1, ni))]
    E = I.random_field(rng, cells, 2e4, dt)
    for sp in (0, 1):
        sim.set_state(0, sp, st[sp])
        ref.set_state(sp, st[sp])

    def same(what):
        assert sim.counters(0) == ref.counters(), what
        for sp in (0, 1):
            a, b = sim.get_state(0, sp), ref.get_state(sp)
            assert a["c"].size == b["c"].size, what
            for k in ("c", "f", "vx", "vy", "vz"):
                assert np.array_equal(a[k], b[k]), (what, sp, k)
            assert np.array_equal(sim.get_deposit(0, sp), ref.get_deposit(sp)), (what, sp)
        assert np.array_equal(sim.get_energy_deposit(0), ref.get_energy_deposit()), what

    for rnd in range(2):
        for n in range(steps):
            sim.set_field(0, E)
            ref.set_field(E)
            sim.sweep()
            ref.sweep()
            same((rnd, n))
        sim.sort()
        ref.sort()
    sim.close()
