"""Rf periods of an odd number of steps, replayed as graphs: the deposits and the voltage scale alternate between
two arrays from solve to solve, so each replay starts in the other one. Single sweeps (whose deposits stay for the
caller), deposits read and set, stand-alone solves and the voltage of the current-driven mode between the replays
give what plain launches give, bit for bit, and the deposits read back hold every particle."""
import math

import numpy as np
import pytest

import inputs as I
from paper_1608_04601_gb300 import xsections as X

pytestmark = pytest.mark.gpu

P = 45  # steps per rf period


def _calls(sim):
    """The sequence of calls; yields everything that it reads."""
    def voltage():
        applied, now = sim.voltage_amplitude(0)
        yield applied
        yield np.asarray(now)

    def deposits():
        for sp in (0, 1):
            D = sim.get_deposit(0, sp)
            yield D
            assert int(D.sum()) == sim.count(0, sp) << 32  # every particle deposits 2^32

    def solved():
        phi, n = sim.get_field(0)[2], sim.step_index
        yield phi
        if n % P:  # at the driven electrode: the present amplitude times the sine at the time of the solve
            V = sim.voltage_amplitude(0)[1]
            assert abs(phi[0] - V * math.sin(2 * math.pi * n / P)) <= 1e-9 * V
        for sp in (0, 1):
            assert not sim.get_deposit(0, sp).any()  # cleared for the next sweep

    sim.step(P)
    yield from voltage()
    sim.step(2 * P)
    yield from voltage()
    yield from solved()
    sim.sweep()
    yield from deposits()
    sim.step(P)  # over the deposits that the single sweep left
    yield from voltage()
    yield from solved()
    sim.sweep()
    D = [sim.get_deposit(0, sp) for sp in (0, 1)]
    for sp in (0, 1):
        sim.set_deposit(0, sp, D[sp][::-1].copy())
    sim.solve()  # the step advances: the replays from here start one step into the period
    yield from solved()
    sim.step(P)
    yield from voltage()
    sim.set_deposit(0, 0, D[0])  # never solved: the next sweep clears it
    sim.step(3 * P + 7)
    yield from voltage()
    yield from solved()
    sim.sweep()
    yield from deposits()
    sim.reset_moments()
    sim.step(2 * P)
    m = sim.moments(0)
    for k in ("n_e", "n_i", "mean_eps", "J_amp", "J_last"):
        yield np.asarray(m[k])
    for sp in (0, 1):
        st = sim.get_state(0, sp)
        for k in ("c", "f", "vx", "vy", "vz"):
            yield st[k]


@pytest.mark.parametrize("sort_every", [0, 5])
@pytest.mark.parametrize("drive", [0.0, 40.0])
def test_replays_of_odd_periods(sort_every, drive):
    import __graft_entry__ as g
    g.build()
    from paper_1608_04601_gb300 import pic
    gas = X.he_like(eps_max_eV=300.0, de_eV=1e-2)
    d = I.discharge(n_cells=129, p_Pa=15.0, V_rf_V=100.0, f_rf_Hz=1e8, n_e0=20001, n_i0=20002, n_init_m3=4e14,
                    gamma_see=0.1, steps_per_period=P)
    got = []
    for graph in (True, False):
        sim = pic.Simulation(gas, d, seed=6, sort_every=sort_every, use_graph=graph, capacity=[(200000, 200000)])
        if drive:
            sim.set_current_drive(0, drive)
        got.append(list(_calls(sim)))
        sim.close()
    assert len(got[0]) == len(got[1])
    for k, (a, b) in enumerate(zip(*got)):
        assert np.array_equal(a, b), k
