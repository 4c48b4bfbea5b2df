"""The mixed kick of systems with a giant planet, whose critical radius is many times the
others' (near tiles take the lo parts in packed pairs): against the oracle's accelerations, with
pairs inside their own radii, coincident bodies, small bodies, counts around the tiles;
and a step in which members' kicks are put right afterwards.

Bound: a term rounds about a dozen times in FP32, 16 x 2^-23 of its magnitude at most; the plain
sums of a 256-body tile's even and odd terms add 128 x 2^-24 of their magnitudes at worst.
"""
import numpy as np
import pytest

import opal_ic as ic

pytestmark = pytest.mark.gpu


def _system(n, n_big):
    s = ic.equal_mass_disk(n, n)
    m, x = s.m.copy(), s.x.copy()
    m[n_big:] = 0.0
    m[n_big // 2] = 1e-3
    x[5] = x[2] + 1e-6          # deep inside both critical radii
    x[n_big - 1] = x[n_big - 2] + 2e-3
    x[n - 1] = x[n_big // 3]    # coincident with a massive body
    return ic.System(f"wide{n}", m, x, s.v, s.R, dt=s.dt, nsteps=2)


@pytest.mark.parametrize("form", [0, 1])
@pytest.mark.parametrize("variant", [0, 3, 4])
@pytest.mark.parametrize("n,n_big", [(1600, 1600), (2049, 300), (2305, 257)])
def test_wide_kick_against_oracle(monkeypatch, n, n_big, variant, form):
    import oracle
    from paper_2601_19654_gb300 import opal
    oracle.build()
    monkeypatch.setenv("OPAL_KICK_VARIANT", str(variant))
    s = _system(n, n_big)
    rc = oracle.hill_rcrit(1.0, 3.0, s.m, s.x)
    with opal.Simulation(s.m, s.x, s.v, s.R, precision=1, changeover=form) as sim:
        a = sim.debug_accel(rc)
    # a coincident pair adds nothing to either; the oracle has no value for it, so each of the
    # two is taken from the system without the other
    want = oracle.accel(1.0, s.m, s.x, rc, form=form)
    for i, other in ((n - 1, n_big // 3), (n_big // 3, n - 1)):
        keep = np.arange(n) != other
        want[i] = oracle.accel(1.0, s.m[keep], s.x[keep], rc[keep], form=form)[i - (other < i)]
    size = np.zeros(n)
    for i in range(0, n, 256):
        d = s.x[None, :, :] - s.x[i:i + 256, None, :]
        r2 = (d * d).sum(2)
        r2[r2 == 0] = np.inf
        size[i:i + 256] = (s.m[None, :] / r2).sum(1)
    assert np.all(np.abs(a - want) <= (16 * 2.0 ** -23 + 128 * 2.0 ** -24) * size[:, None])


@pytest.mark.parametrize("order", ["overlap", "inorder"])
def test_wide_step_against_oracle(monkeypatch, order):
    """Both orders of the step (the one beside the encounters patches members' terms)."""
    import oracle
    from paper_2601_19654_gb300 import opal
    oracle.build()
    monkeypatch.setenv("OPAL_STEP_ORDER", order)
    s = ic.planetesimals_jupiter(4, 2500)
    osim = oracle.Sim.from_system(s)
    assert osim.step(2) == oracle.OK
    alive = np.nonzero(osim.alive)[0]
    with opal.Simulation.from_system(s, precision=1) as sim:
        sim.step(2)
        assert sim.step_overlap == (order == "overlap")
        assert sim.stats()["n_groups"] > 0
        st = sim.state()
    assert st["ids"].tolist() == alive.tolist()
    err = np.linalg.norm(st["x"] - osim.x[alive], axis=1) / np.linalg.norm(osim.x[alive], axis=1)
    assert err.max() <= 1e-6, err.max()      # (the mixed form's bound elsewhere)
