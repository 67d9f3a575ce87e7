"""The sweep where a CTA flushes its histograms in the middle of a store and goes on with it, bit for bit against
the oracle: state, order, counters, deposits and energy moment.

A CTA adds at most 32768 particles of a store in FP32 (16384 in FP64) between flushes, so with one CTA per SM
the stores here, of more than 5e6 (2.6e6) particles, cross a flush on a GPU of up to 152 SMs. They end in the
middle of a row. Sorted stores with windows, one with a cell range beyond a window's; one histogram set (4096
cells); and the largest sums a piece may hold: every particle of the store in one cell at an offset next to 1,
electrons just below 32 eV (17 set bits of energy in the low piece) and beyond the clamp at 16384 eV. Then
batches whose CTAs go from one discharge to the next with windows, with two histogram sets and with one."""
import numpy as np
import pytest

import inputs as I
from oracle import oracle as O
from paper_1608_04601_gb300 import xsections as X

pytestmark = pytest.mark.gpu

KEYS = ("c", "f", "vx", "vy", "vz")


@pytest.fixture(scope="module")
def P():
    import __graft_entry__ as g
    g.build()
    from paper_1608_04601_gb300 import pic
    return pic


def _store(rng, kind, n, cells, sp, dt, d):
    if kind == "mixed":
        return I.mixed_state(rng, n, cells, sp, dt, d.gap_m, d.dt_s)
    f = np.nextafter(dt(1), dt(0))
    st = {"c": np.full(n, cells // 2, np.int32), "f": np.full(n, f, dt)}
    eV = 20000.0 if kind == "beyond clamp" else 32.0 - 1.5 * 2.0**-12
    v = np.sqrt(2 * I.E_CH * eV / I.M_E) if sp == 0 else 0.0
    for k in ("vx", "vy", "vz"):
        st[k] = np.full(n, v if k == "vx" else 0.0, dt)
    return st


def _same(sim, i, ref, what):
    assert sim.counters(i) == ref.counters(), what
    for sp in (0, 1):
        assert np.array_equal(sim.get_deposit(i, sp), ref.get_deposit(sp)), (what, sp)
        a, b = sim.get_state(i, sp), ref.get_state(sp)
        for k in KEYS:
            assert np.array_equal(a[k], b[k]), (what, sp, k)
    assert np.array_equal(sim.get_energy_deposit(i), ref.get_energy_deposit()), what


def _run(P, prec, specs, steps):
    """specs: (kind, cells, electrons, ions) of each discharge."""
    dt = np.float32 if prec == "fp32" else np.float64
    gas = X.he_like(eps_max_eV=200.0, de_eV=1e-2)
    rng = np.random.default_rng(len(specs) + specs[0][1])
    ds = [I.discharge(n_cells=N, p_Pa=100.0 if kind == "mixed" else 1e-3, gamma_see=0.2, V_rf_V=100.0, seed=3,
                      discharge_id=i) for i, (kind, N, _, _) in enumerate(specs)]
    caps = [(a + a // 8 + 40000, b + a // 8 + 40000) for _, _, a, b in specs]
    sim = P.Simulation(gas, ds, seed=3, precision=prec, load=False, capacity=caps)
    refs, fields = [], []
    for i, (kind, N, a, b) in enumerate(specs):
        refs.append(O.Oracle(gas, ds[i], "f32" if prec == "fp32" else "f64", load=False))
        fields.append(I.random_field(rng, N, 2e4 if kind == "mixed" else 0.0, dt))
        for sp, n in ((0, a), (1, b)):
            st = _store(rng, kind, n, N, sp, dt, ds[i])
            sim.set_state(i, sp, st)
            refs[i].set_state(sp, st)
    for s in range(steps):
        for i in range(len(specs)):
            sim.set_field(i, fields[i])
            refs[i].set_field(fields[i])
            refs[i].sweep()
        sim.sweep()
        for i in range(len(specs)):
            _same(sim, i, refs[i], (s, i))
    sim.close()


@pytest.mark.parametrize("prec,kind,cells,n", [
    ("fp32", "mixed", 512, 5_300_003), ("fp32", "mixed", 40, 5_200_017), ("fp32", "mixed", 4096, 5_100_011),
    ("fp32", "below 32 eV", 100, 5_100_011), ("fp32", "beyond clamp", 100, 5_100_011),
    ("fp64", "mixed", 512, 2_700_005), ("fp64", "below 32 eV", 100, 2_600_011), ("fp64", "beyond clamp", 100, 2_600_011)])
def test_flush_within_a_store(P, prec, kind, cells, n):
    _run(P, prec, [(kind, cells, n, n - 100_003 if kind == "mixed" else n)], 1)


@pytest.mark.parametrize("prec,cells", [("fp32", (512, 201, 512)), ("fp32", (3500, 4096, 800)), ("fp64", (512, 201, 512)),
                                        ("fp64", (4096, 3100, 64))])
def test_batches_with_windows(P, prec, cells):
    sizes = [(450_007, 400_009), (500_021, 520_003), (380_001, 390_013)]
    _run(P, prec, [("mixed", N, a, b) for N, (a, b) in zip(cells, sizes)], 2)
