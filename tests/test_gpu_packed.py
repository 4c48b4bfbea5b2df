"""More groups in a step than the lockstep kernels take (4864): close pairs and triples of one
system through the packed kernel, with the larger chance groups beside it, against the oracle.

Tolerance: 1e-9 of a position, as for the encounter kernels elsewhere.
"""
import numpy as np
import pytest

import opal_ic as ic

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("groups,triples,precision,tol", [(5400, 0, 0, 1e-9), (5200, 1500, 0, 1e-9), (5400, 300, 1, 1e-6)])
def test_many_small_groups_match_the_oracle(groups, triples, precision, tol):
    import oracle
    from paper_2601_19654_gb300 import opal
    oracle.build()
    rng = np.random.default_rng(groups + triples)
    s = ic.equal_mass_disk(3, groups)
    rc = 3.0 * np.linalg.norm(s.x, axis=1) * np.cbrt(s.m / 3.0)
    parts = [(s.x, s.v)]
    for k, count in ((0, groups), (1, triples)):
        u = rng.normal(size=(count, 3))
        u *= (rng.uniform(0.3, 0.9, count) * rc[:count] / np.linalg.norm(u, axis=1))[:, None]
        parts.append((s.x[:count] + u, s.v[:count] * (1.0 + 1e-4 * rng.normal(size=(count, 1)))))
    x, v = np.concatenate([p[0] for p in parts]), np.concatenate([p[1] for p in parts])
    n = len(x)
    sysm = ic.System("pairs", np.full(n, s.m[0]), x, v, np.full(n, s.R[0] * 1e-2), dt=s.dt * 0.5, nsteps=1)
    osim = oracle.Sim.from_system(sysm, scan_prune=1)
    assert osim.step(1) == oracle.OK
    alive = np.nonzero(osim.alive)[0]
    with opal.Simulation.from_system(sysm, precision=precision) as sim:
        sim.step(1)
        assert sim.stats()["n_groups"] > 4864
        st = sim.state()
    assert st["ids"].tolist() == alive.tolist()
    err = np.linalg.norm(st["x"] - osim.x[alive], axis=1) / np.linalg.norm(osim.x[alive], axis=1)
    assert err.max() <= tol, err.max()


def _crowd(massless, touching):
    """5400 primaries of a disk, each with a close companion, the first 600 with a third body: the companions
    massive, the last of them, or all, massless; radii small, or such that about a third of the pairs touch."""
    rng = np.random.default_rng(17 + 2 * massless + touching)
    groups, triples = 5400, 600
    s = ic.equal_mass_disk(3, groups)
    rc = 3.0 * np.linalg.norm(s.x, axis=1) * np.cbrt(s.m / 3.0)

    def near(k):
        u = rng.normal(size=(len(k), 3))
        u *= (rng.uniform(0.3, 0.9, len(k)) * rc[k] / np.linalg.norm(u, axis=1))[:, None]
        return s.x[k] + u, s.v[k] * (1.0 + 1e-4 * rng.normal(size=(len(k), 1)))
    k = np.concatenate([np.arange(groups), np.arange(groups), np.arange(triples)])
    xv = [(s.x, s.v), near(np.arange(groups)), near(np.arange(triples))]
    x, v = np.concatenate([p[0] for p in xv]), np.concatenate([p[1] for p in xv])
    m = np.full(len(x), s.m[0])
    # (a system's massless bodies come last): the third bodies and the companions of the later primaries, or all companions
    m[groups if massless == 2 else groups + 2000:] = 0.0 if massless else s.m[0]
    R = np.where(touching, 0.25, 1e-3) * rc[k]
    return ic.System("crowd", m, x, v, R, dt=s.dt * 0.5, nsteps=1)


@pytest.mark.parametrize("massless,touching", [(0, True), (1, False), (1, True), (2, False), (2, True)])
def test_mergers_and_massless_members_match_the_oracle(massless, touching):
    """The packed kernel's mergers and its members that pull nothing."""
    import oracle
    from paper_2601_19654_gb300 import opal
    oracle.build()
    s = _crowd(massless, touching)
    osim = oracle.Sim.from_system(s, scan_prune=1)
    assert osim.step(1) == oracle.OK
    alive = np.nonzero(osim.alive)[0]
    assert (s.n - alive.size > 1000) == touching
    with opal.Simulation.from_system(s, precision=0) as sim:
        sim.step(1)
        stats = sim.stats()
        assert stats["n_groups"] > 4864 and stats["n_mergers"] == s.n - alive.size
        st = sim.state()
    assert st["ids"].tolist() == alive.tolist()
    err = np.linalg.norm(st["x"] - osim.x[alive], axis=1) / np.linalg.norm(osim.x[alive], axis=1)
    assert err.max() <= 1e-9, err.max()
    np.testing.assert_allclose(st["m"], osim.m[alive], rtol=1e-14, atol=0)
    np.testing.assert_allclose(st["R"], osim.R[alive], rtol=1e-14, atol=0)
