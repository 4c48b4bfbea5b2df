"""One small system's step (scan and groups in one kernel, the mixed kick a warp a body)
against the general kernels, which the same system twice in one simulation takes, and
against the oracle's accelerations; counts around the tile and warp edges and at the
largest size of that path.

Bounds: a mixed pair term rounds about a dozen times in FP32 (separation, its square,
1/r^3, the product with the mass), 16 x 2^-23 of its magnitude at most; velocities after a
step differ by the two kicks of dt / 2 and the rounding of FP64, 1e-12.  A member of an encounter
group carries the opening kick's difference through the encounter: it is held to 1e-5 only.
"""
import numpy as np
import pytest

import opal_ic as ic

pytestmark = pytest.mark.gpu

MIXED_TERM = 16 * 2.0 ** -23
SIZES = [(1, 1), (2, 2), (5, 5), (10, 1), (33, 32), (64, 64), (65, 65), (257, 129), (513, 512), (1001, 1001),
         (1536, 1500)]


def _system(n, n_big):
    s = ic.equal_mass_disk(n + 7, n)
    m, x = s.m * 50.0, s.x.copy()
    m[n_big:] = 0.0
    if n_big > 3:
        m[n_big // 2] = 1e-3
    if n > 8:
        x[5] = x[2] + 1e-6      # deep inside both critical radii
    return m, x, s.v, s.R


def _size(m, x):
    d = x[None, :, :] - x[:, None, :]
    r2 = (d * d).sum(2)
    r2[r2 == 0] = np.inf
    return (m[None, :] / r2).sum(1)


@pytest.mark.parametrize("form", [0, 1])
@pytest.mark.parametrize("n,n_big", SIZES)
def test_small_mixed_kick_against_oracle(n, n_big, form):
    import oracle
    from paper_2601_19654_gb300 import opal
    oracle.build()
    m, x, v, R = _system(n, n_big)
    rc = oracle.hill_rcrit(1.0, 3.0, m, x)
    with opal.Simulation(m, x, v, R, precision=1, changeover=form) as sim:
        a = sim.debug_accel(rc)
    want = oracle.accel(1.0, m, x, rc, form=form)
    assert np.all(np.abs(a - want) <= MIXED_TERM * _size(m, x)[:, None])


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("n,n_big", SIZES)
def test_small_scan_and_step_against_general(n, n_big, precision):
    from paper_2601_19654_gb300 import opal
    m, x, v, R = _system(n, n_big)
    dt = 0.01
    two = lambda a: np.concatenate([a, a])
    with opal.Simulation(m, x, v, R, precision=precision, dt=dt) as sim, \
            opal.Simulation(two(m), two(x), two(v), two(R), n_per_sys=[n, n], precision=precision, dt=dt) as ref:
        # the scan alone: start and end of a drift, critical radii that flag many pairs
        x1, v1 = opal.debug_drift(1.0, dt, x, v)[:2]
        rc = np.random.default_rng(n).uniform(0.0, 40.0 / n, n)
        i, j, cand = sim.debug_scan(x, v, x1, v1, rc)
        gi, gj, gcand = ref.debug_scan(two(x), two(v), two(x1), two(v1), two(rc))
        one = gi < n
        assert np.array_equal(np.stack([i, j]), np.stack([gi[one], gj[one]]))
        assert np.array_equal(gi[one] + n, gi[~one]) and 2 * cand == gcand
    with opal.Simulation(m, x, v, R, precision=precision, dt=dt) as sim, \
            opal.Simulation(two(m), two(x), two(v), two(R), n_per_sys=[n, n], precision=precision, dt=dt) as ref:
        sim.step(1)
        ref.step(1)
        a, b = sim.stats(), ref.stats()
        for k in ("n_pairs", "n_groups", "n_mergers", "n_candidates"):
            assert 2 * a[k] == b[k], k
        s, r = sim.state(), ref.state(1)
    assert s["m"].size == r["m"].size
    np.testing.assert_allclose(s["m"], r["m"], rtol=1e-14)
    if s["m"].size != n:
        return                  # a merger: the bodies' order is no longer the input's
    term = MIXED_TERM if precision == 1 else 2.0 ** -47
    tol = dt * term * _size(m, x) + 1e-12 * np.linalg.norm(v, axis=1)
    if a["n_groups"]:
        rcm = 3.0 * np.linalg.norm(x, axis=1) * np.cbrt(m / 3.0)
        d = np.linalg.norm(x[None] - x[:, None], axis=2) + 2 * np.eye(n)
        near = d < np.maximum(rcm[None], rcm[:, None]) + 4 * dt * np.linalg.norm(v, axis=1).max()
        tol = np.where(near.any(1), 1e-5 * np.linalg.norm(v, axis=1), tol)
    assert np.all(np.linalg.norm(s["v"] - r["v"], axis=1) <= tol)
    assert np.all(np.linalg.norm(s["x"] - r["x"], axis=1) <= dt * tol + 1e-12)


def test_the_kick_named_is_the_one_that_runs(monkeypatch):
    from paper_2601_19654_gb300 import opal
    m, x, v, R = _system(500, 500)
    with opal.Simulation(m, x, v, R, precision=1, dt=0.01) as sim:
        for order, tiled in (("inorder", False), ("overlap", True), (None, False)):
            if order:
                monkeypatch.setenv("OPAL_STEP_ORDER", order)
            else:
                monkeypatch.delenv("OPAL_STEP_ORDER")
            sim.step(1)
            assert sim.step_overlap == tiled
            assert sim.kick_config.startswith("mixed t" if tiled else "mixed, a warp a body")


# A body so far away that the float square of a separation overflows (beyond 1.8e19), massive or not:
# it pulls nothing that a float holds, and the others' accelerations are as without it.
@pytest.mark.parametrize("massive", [True, False])
@pytest.mark.parametrize("far", [1e18, 1e20, 1e30])
def test_a_body_beyond_the_float_squares(far, massive):
    from paper_2601_19654_gb300 import opal
    m, x, v, R = _system(40, 40)
    m[-1] = m[-1] if massive else 0.0
    x[-1], v[-1] = [far, 0.0, 0.0], [0.0, far ** -0.5, 0.0]
    with opal.Simulation(m, x, v, R, precision=1, dt=0.01) as sim, \
            opal.Simulation(m[:-1], x[:-1], v[:-1], R[:-1], precision=1, dt=0.01) as ref:
        a, b = sim.debug_accel(), ref.debug_accel()
        assert np.array_equal(a[:-1], b)
        assert np.all(np.abs(a[-1]) <= m.sum() / far ** 2)
        sim.step(1)
        ref.step(1)
        s, r = sim.state(), ref.state()
    assert s["ids"].tolist() == r["ids"].tolist() + [39]   # (two of the others merge)
    # (the barycentre's motion takes the far body's momentum: below 1e-5 x its 1e-9 of a velocity)
    np.testing.assert_allclose(s["x"][:-1], r["x"], rtol=0, atol=1e-12)
