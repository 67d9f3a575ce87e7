"""pic_sort against a stable argsort: stores at the edges of its tiles (4096 slots) and of several tiles,
chunk shapes, odd cell counts, sorted, reversed, uniform and single-cell stores, batches of uneven and empty
stores; after a sweep, so that the sort walks a region layout too."""
import numpy as np
import pytest

import inputs as I
from paper_1608_04601_gb300 import xsections as X

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    import __graft_entry__ as g
    g.build()
    from paper_1608_04601_gb300 import pic
    return pic


def _store(rng, n, cells, kind, dt):
    c = rng.integers(0, cells, n).astype(np.int32)
    if kind == "near":
        c = np.clip(np.sort(c) + rng.integers(-2, 3, n), 0, cells - 1).astype(np.int32)
    elif kind == "reversed":
        c = np.sort(c)[::-1].astype(np.int32)
    elif kind == "one":
        c[:] = cells - 1
    st = {"c": c, "f": rng.uniform(0, 0.99, n).astype(dt)}
    for k in ("vx", "vy", "vz"):
        st[k] = rng.normal(0, 1e3, n).astype(dt)
    return st


def _check(sim, d):
    for sp in (0, 1):
        a = sim.get_state(d, sp)
        order = np.argsort(a["c"], kind="stable")
        yield sp, {k: v[order] for k, v in a.items()}


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
@pytest.mark.parametrize("cells,ppt,sizes,kind", [
    (128, 4, [(20000, 33000)], "near"), (1, 4, [(32768, 32769)], "one"), (333, 2, [(32767, 4097)], "uniform"),
    (512, 8, [(100001, 31)], "reversed"), (4096, 4, [(70000, 12345)], "near"), (97, 4, [(0, 1)], "one"),
    (64, 4, [(1000, 50000), (32768, 40000), (0, 0), (90001, 2)], "near"), (2047, 2, [(250000, 40000)], "uniform")])
def test_sort_is_stable(P, prec, cells, ppt, sizes, kind):
    rng = np.random.default_rng(cells + ppt)
    dt = np.float32 if prec == "fp32" else np.float64
    gas = X.he_like(eps_max_eV=100.0, de_eV=1e-2)
    ds = [I.discharge(n_cells=cells, n_e0=1, n_i0=1, discharge_id=i) for i in range(len(sizes))]
    sim = P.Simulation(gas, ds, precision=prec, load=False, ppt=ppt, capacity=[(2 * a + 5000, 2 * b + 5000) for a, b in sizes])
    for d, (a, b) in enumerate(sizes):
        for sp, n in ((0, a), (1, b)):
            sim.set_state(d, sp, _store(rng, n, cells, kind, dt))
    for after_sweep in (False, True):
        if after_sweep:
            sim.sweep()
        want = [list(_check(sim, d)) for d in range(len(ds))]
        sim.sort()
        for d in range(len(ds)):
            for sp, w in want[d]:
                got = sim.get_state(d, sp)
                for k in w:
                    assert np.array_equal(got[k], w[k]), (after_sweep, d, sp, k)
    sim.close()
