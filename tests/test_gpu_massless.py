"""Simulations in which no body has mass (test particles about the star): every body follows its own
Kepler orbit, in both forms, in systems of the small path, of the general one and in an ensemble with
an empty-handed system beside a massive one.

Tolerance: 1e-12 of a position against the oracle's drift, as for a lone test mass.
"""
import numpy as np
import pytest

import opal_ic as ic

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("n", [1, 40, 2000])
def test_massless_bodies_follow_their_orbits(n, precision):
    import oracle
    from paper_2601_19654_gb300 import opal
    oracle.build()
    d = ic.equal_mass_disk(3, n)
    s = ic.System("massless", np.zeros(n), d.x, d.v, np.zeros(n), dt=0.05, nsteps=3)
    osim = oracle.Sim.from_system(s)
    assert osim.step(3) == oracle.OK
    with opal.Simulation.from_system(s, precision=precision) as sim:
        sim.step(3)
        st = sim.state()
        E, L, P, lost = sim.energy()
        assert sim.stats()["n_pairs"] == 0
    assert st["ids"].size == n
    err = np.linalg.norm(st["x"] - osim.x, axis=1) / np.linalg.norm(osim.x, axis=1)
    assert err.max() <= 1e-12, err.max()
    assert E == 0.0 and lost == 0.0 and not L.any() and not P.any()


@pytest.mark.parametrize("precision", [0, 1])
def test_massless_system_beside_a_massive_one(precision):
    from paper_2601_19654_gb300 import opal
    a, d = ic.equal_mass_disk(4, 300), ic.equal_mass_disk(5, 200)
    b = ic.System("massless", np.zeros(200), d.x, d.v, np.zeros(200), dt=a.dt, nsteps=2)
    with opal.Simulation.from_system(b, precision=precision) as one, \
            opal.Simulation.ensemble([a, b], precision=precision) as both:
        one.step(2)
        both.step(2)
        np.testing.assert_allclose(both.state(1)["x"], one.state()["x"], rtol=0, atol=1e-14)
