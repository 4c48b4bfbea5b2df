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
