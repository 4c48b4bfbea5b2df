"""The state's copy out, by size: one block, a cluster, and two kernels with copies straight to
the caller; sizes around the lines between them, with every body alive, with bodies
scattered over the system gone, and with all of them gone but one; any array left out.

Positions come back as they went in; a velocity goes through the democratic heliocentric frame
and back, two roundings of a number of the size of the momentum sum over M0.
"""
import ctypes as C

import numpy as np
import pytest

import opal_ic as ic

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 2, 255, 256, 257, 1281, 2000, 8192, 8193, 20001])
def test_state_returns_the_bodies(n):
    from paper_2601_19654_gb300 import opal
    s = ic.equal_mass_disk(n, n)
    with opal.Simulation.from_system(s, precision=1) as sim:
        st = sim.state()
        again = sim.state()
    assert st["ids"].tolist() == list(range(n))
    for k, want in (("m", s.m), ("x", s.x), ("R", s.R)):
        assert np.array_equal(st[k], want), k
    np.testing.assert_allclose(st["v"], s.v, rtol=0, atol=1e-15)
    assert all(np.array_equal(st[k], again[k]) for k in st)


@pytest.mark.parametrize("n", [5, 257, 1281, 8192, 8193, 20001])
@pytest.mark.parametrize("keep", ["some", "one"])
def test_state_after_removals(n, keep):
    from paper_2601_19654_gb300 import opal
    rng = np.random.default_rng(n)
    s = ic.equal_mass_disk(n, n)
    gone = rng.random(n) < (0.3 if keep == "some" else 2.0)
    gone[n // 2] = False
    x = np.where(gone[:, None], s.x * (100.0 / np.linalg.norm(s.x, axis=1))[:, None], s.x)
    v = np.where(gone[:, None], s.v * 0.05, s.v)
    m = s.m * 1e-3
    with opal.Simulation(m, x, v, s.R * 1e-3, precision=1, dt=1e-3, r_eject=50.0, eject_every=1) as sim:
        sim.step(1)
        st = sim.state()
        buf_x, buf_v = np.full((n, 3), 7.0), np.full((n, 3), 7.0)
        na = C.c_int64(0)
        L = opal.lib()
        raw = C.CDLL(L._name).opal_get_state
        raw.restype = C.c_int32
        p = lambda a: None if a is None else C.c_void_p(a.ctypes.data)
        raw.argtypes = [C.c_void_p, C.c_int32, C.c_void_p] + [C.c_void_p] * 5
        # some of the arrays only; nothing is written past the live bodies
        assert raw(sim.ptr, 0, C.byref(na), None, None, p(buf_x), p(buf_v), None) == 0
    ids = np.nonzero(~gone)[0]
    assert st["ids"].tolist() == ids.tolist() and na.value == ids.size
    assert np.array_equal(st["m"], m[ids]) and np.array_equal(st["R"], (s.R * 1e-3)[ids])
    step = 1e-3 * (np.linalg.norm(v[ids], axis=1) + 0.1)
    assert np.all(np.linalg.norm(st["x"] - x[ids], axis=1) <= step)
    assert np.array_equal(buf_x[:ids.size], st["x"]) and np.array_equal(buf_v[:ids.size], st["v"])
    assert np.all(buf_x[ids.size:] == 7.0) and np.all(buf_v[ids.size:] == 7.0)
