"""Upload of a store at sizes around the pack kernel's edges (16-byte groups, a CTA's threads, several
CTAs): the last CTA sets count and layout and passes the check word on, from pinned arrays and through
staging; a cell out of range anywhere leaves an empty store, and the next upload is not affected. The
combined read-backs (moments, field) agree with the single ones."""
import numpy as np
import pytest

import inputs as I
from paper_1608_04601_gb300 import xsections as X

pytestmark = pytest.mark.gpu

KEYS = ("c", "f", "vx", "vy", "vz")


@pytest.fixture(scope="module")
def P():
    import __graft_entry__ as g
    g.build()
    from paper_1608_04601_gb300 import pic
    return pic


@pytest.fixture(scope="module", params=["fp32", "fp64"])
def sim(P, request):
    d = I.discharge(n_cells=101, gap_m=0.025, p_Pa=60.0, V_rf_V=300.0, n_e0=5000, n_i0=5000, n_init_m3=4e14)
    s = P.Simulation(X.he_like(eps_max_eV=600.0, de_eV=1e-2), d, precision=request.param, capacity=[(250_000, 250_000)])
    yield s
    s.close()


def _state(n, N, dt, pinned, seed):
    import torch
    rng = np.random.default_rng(seed)
    st = {}
    for k in KEYS:
        a = rng.integers(0, N, n).astype(np.int32) if k == "c" else rng.random(n).astype(dt)
        st[k] = torch.from_numpy(a).pin_memory().numpy() if pinned else a
    return st


@pytest.mark.parametrize("pinned", [True, False])
@pytest.mark.parametrize("n", [0, 1, 3, 4, 5, 1023, 1025, 200_003])
def test_upload_edges(P, sim, n, pinned):
    from paper_1608_04601_gb300 import _native as NV
    dt, N = np.dtype(sim.dtype), sim.N[0]
    st = _state(n, N, dt, pinned, n)
    if n:
        for at, cell in ((0, -1), (n - 1, N), (n // 2, 2**31 - 1)):
            keep = int(st["c"][at])
            st["c"][at] = cell
            with pytest.raises(NV.PicError):
                sim.set_state(0, 1, st)
            st["c"][at] = keep
            assert sim.count(0, 1) == 0
    sim.set_state(0, 1, st)
    got = sim.get_state(0, 1)
    assert sim.count(0, 1) == n and all(np.array_equal(got[k], st[k]) for k in KEYS)
    out = _state(n + 3, N, dt, True, 1)
    got = sim.get_state(0, 1, out=out)
    assert all(np.array_equal(got[k], st[k]) for k in KEYS)


def test_combined_readbacks(sim):
    sim.step(3)
    m = sim.moments(0)
    assert m["count"] == [sim.count(0, 0), sim.count(0, 1)]
    assert m["J_last"] == sim.current(0, 2, 1)[0, 0]
    E, E64, phi = sim.get_field(0)
    assert phi.size == sim.N[0] + 1
    np.testing.assert_allclose(E, E64, rtol=2.0**-23)  # the FP32 field is the FP64 one, rounded
    E[:] = np.arange(E.size)
    sim.set_field(0, E)
    assert np.array_equal(sim.get_field(0)[0], E)
