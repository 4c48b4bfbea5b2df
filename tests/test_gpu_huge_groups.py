"""Encounter groups of more than 64 members, by what bounds them: everyone near everyone
(few members to a warp, no lists), a few near ones each (lists of fewer members to a
warp), one giant among massive and massless bodies, and more wide members than a
block keeps copies of; with and without mergers; one step against the oracle.

Tolerance: 1e-9 of a position, as for the other groups of this size (an accept decision
of a group of hundreds can sit within rounding of the encounter tolerance, 1e-12 of the state).
"""
import numpy as np
import pytest

import opal_ic as ic

pytestmark = pytest.mark.gpu


def _cloud(seed, n, at, v, spread, vspread):
    rng = np.random.default_rng(seed)
    x = np.array([at, 0.0, 0.0]) + rng.normal(0.0, spread, (n, 3))
    return x, np.array([0.0, v, 0.0]) + rng.normal(0.0, vspread, (n, 3))


def _dense(n, R):
    x, v = _cloud(n, n, 1.0, 1.0, 2e-3, 1e-3)
    return ic.System(f"dense{n}", np.full(n, 1e-8), x, v, np.full(n, R), dt=0.02, nsteps=1)


def _middling(n):
    x, v = _cloud(7, n, 1.0, 1.0, 6e-3, 1e-3)
    return ic.System(f"middling{n}", np.full(n, 1e-8), x, v, np.full(n, 2e-6), dt=0.02, nsteps=1)


def _giant(n, n_big, R):
    x, v = _cloud(5, n, 5.0, 0.447, 0.1, 5e-3)
    m = np.zeros(n)
    m[0], m[1:n_big] = 1e-3, 1e-9
    x[0] = [5.0, 0.0, 0.0]
    r = np.full(n, R)
    r[0] = 4e-4
    return ic.System(f"giant{n}", m, x, v, r, dt=0.1, nsteps=1)


def _many_wide(n, wide):
    x, v = _cloud(9, n, 5.0, 0.447, 0.1, 5e-3)
    m = np.full(n, 1e-10)
    m[:wide] = 1e-5
    return ic.System(f"wide{wide}", m, x, v, np.full(n, 1e-6), dt=0.02, nsteps=1)


@pytest.mark.parametrize("make,merges", [
    (lambda: _dense(65, 1e-6), False), (lambda: _dense(150, 2e-4), True), (lambda: _middling(600), False),
    (lambda: _giant(300, 40, 1e-6), False), (lambda: _giant(129, 129, 3e-4), True),
    (lambda: _many_wide(200, 3), False), (lambda: _many_wide(200, 18), False),
])
def test_one_step_of_a_large_group_against_oracle(make, merges):
    import oracle
    from paper_2601_19654_gb300 import opal
    oracle.build()
    s = make()
    osim = oracle.Sim.from_system(s, scan_prune=1)
    assert osim.step(1) == oracle.OK
    alive = np.nonzero(osim.alive)[0]
    assert (alive.size < s.n) or not merges
    states = []
    for _ in range(2):
        with opal.Simulation.from_system(s, precision=0, encounter_capacity=1 << 17) as sim:
            sim.step(1)
            states.append(sim.state())
    a, b = states
    assert np.array_equal(a["x"], b["x"]) and np.array_equal(a["v"], b["v"])   # the same on every run
    assert a["ids"].tolist() == alive.tolist()
    err = np.linalg.norm(a["x"] - osim.x[alive], axis=1) / np.linalg.norm(osim.x[alive], axis=1)
    assert err.max() <= 1e-9, err.max()
    np.testing.assert_allclose(a["m"], osim.m[alive], rtol=1e-14, atol=0)


# A dense group alone takes the blocks of both teams, a member a warp in its last rounds
# (700 and 1000 warps, more than a group with lists ever has); a short step, of few substeps.
@pytest.mark.parametrize("n", [700, 1000])
def test_dense_group_of_a_member_a_warp(n):
    import oracle
    from paper_2601_19654_gb300 import opal
    oracle.build()
    x, v = _cloud(n, n, 1.0, 1.0, 2e-3, 1e-3)
    s = ic.System(f"dense{n}", np.full(n, 1e-8), x, v, np.full(n, 1e-9), dt=1e-3, nsteps=1)
    osim = oracle.Sim.from_system(s, scan_prune=1)
    assert osim.step(1) == oracle.OK
    assert osim.alive.all()
    with opal.Simulation.from_system(s, precision=0, encounter_capacity=1 << 20) as sim:
        sim.step(1)
        assert sim.stats()["n_groups"] == 1
        st = sim.state()
    err = np.linalg.norm(st["x"] - osim.x, axis=1) / np.linalg.norm(osim.x, axis=1)
    assert err.max() <= 1e-9, err.max()
