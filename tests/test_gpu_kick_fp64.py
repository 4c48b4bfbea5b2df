"""The FP64 kick's tiles: counts around the tile edges, small bodies, super-tiles,
uneven ensembles, both changeovers, against the oracle's accelerations.

Bound: each term's separation, 1/r^3 and product round at most a dozen times (2^-53
each; near pairs, with the changeover's divisions, about twice that), and a body's sum
of n terms adds at most log-many roundings of its rows and 32 of a run, so each
component is within 64 x 2^-53 of the sum of the terms' magnitudes (inside the 1e-13 of
one stage).
"""
import numpy as np
import pytest

import opal_ic as ic

pytestmark = pytest.mark.gpu


def _system(n, n_big):
    """n bodies, the first n_big with mass: a disk in which near pairs are common,
    with one giant (whose critical radius covers many of the others)."""
    s = ic.equal_mass_disk(n, n)
    m, x = s.m * 50.0, s.x.copy()
    m[n_big:] = 0.0
    if n_big > 3:
        m[n_big // 2] = 1e-3
    if n > 8:
        x[5] = x[2] + 1e-6      # deep inside both critical radii
    return m, x, s.v, s.R


def _check(a, m, x, rc, form):
    import oracle
    want = oracle.accel(1.0, m, x, rc, form=form)
    size = np.zeros(len(m))
    for i in range(0, len(m), 256):
        d = x[None, :, :] - x[i:i + 256, None, :]
        r2 = (d * d).sum(2)
        r2[r2 == 0] = np.inf
        size[i:i + 256] = (m[None, :] / r2).sum(1)
    assert np.all(np.abs(a - want) <= 64 * 2.0 ** -53 * size[:, None])


@pytest.mark.parametrize("variant", [0, 1, 2])
@pytest.mark.parametrize("n,n_big", [(1, 1), (2, 2), (31, 31), (33, 32), (64, 1), (129, 129), (300, 37), (1001, 1001),
                                     (4200, 4129)])
def test_fp64_kick_tiles(monkeypatch, variant, n, n_big):
    import oracle
    from paper_2601_19654_gb300 import opal
    oracle.build()
    monkeypatch.setenv("OPAL_KICK_VARIANT", str(variant))
    m, x, v, R = _system(n, n_big)
    rc = oracle.hill_rcrit(1.0, 3.0, m, x)
    for form in (0, 1):
        with opal.Simulation(m, x, v, R, precision=0, changeover=form) as sim:
            assert sim.kick_config.startswith(f"fp64 w{(1, 2, 4)[variant]}")
            _check(sim.debug_accel(rc), m, x, rc, form)


def test_fp64_kick_uneven_ensemble():
    import oracle
    from paper_2601_19654_gb300 import opal
    oracle.build()
    parts = [_system(n, b) for n, b in ((3, 3), (260, 200), (1, 1), (65, 65), (40, 0), (513, 500))]
    cat = [np.concatenate([p[k] for p in parts]) for k in range(4)]
    rcs = [oracle.hill_rcrit(1.0, 3.0, p[0], p[1]) for p in parts]
    with opal.Simulation(*cat, precision=0, n_per_sys=[len(p[0]) for p in parts]) as sim:
        a = sim.debug_accel(np.concatenate(rcs))
    k = 0
    for p, rc in zip(parts, rcs):
        _check(a[k:k + len(rc)], p[0], p[1], rc, 0)
        k += len(rc)


@pytest.mark.parametrize("n,n_big", [(1, 1), (2, 2), (17, 16), (31, 31), (33, 32), (64, 1), (65, 33), (129, 129),
                                     (300, 37), (900, 900), (700, 200)])
def test_fp64_kick_few_items(n, n_big):
    """Few items: eight warps share an item's steps, steps without a pair left out."""
    import oracle
    from paper_2601_19654_gb300 import opal
    oracle.build()
    m, x, v, R = _system(n, n_big)
    rc = oracle.hill_rcrit(1.0, 3.0, m, x)
    for form in (0, 1):
        with opal.Simulation(m, x, v, R, precision=0, changeover=form) as sim:
            assert sim.kick_config.startswith("fp64 split")
            _check(sim.debug_accel(rc), m, x, rc, form)


# Two massive bodies whose squared separation overflows (and whose own squares do not): the pair
# adds nothing, as 1/r^3 is 0, and the others' accelerations are as without the two.
@pytest.mark.parametrize("variant", [0, 1, 2, None])
def test_fp64_kick_where_a_square_overflows(monkeypatch, variant):
    from paper_2601_19654_gb300 import opal
    if variant is not None:
        monkeypatch.setenv("OPAL_KICK_VARIANT", str(variant))
    m, x, v, R = _system(140, 140)
    far = np.arange(140) >= 138
    x[138], x[139], v[far] = [7e153, 0.0, 0.0], [-7e153, 0.0, 0.0], 0.0
    with opal.Simulation(m, x, v, R, precision=0) as sim, \
            opal.Simulation(m[~far], x[~far], v[~far], R[~far], precision=0) as ref:
        a, b = sim.debug_accel(), ref.debug_accel()
    assert not a[far].any()
    np.testing.assert_allclose(a[~far], b, rtol=0, atol=1e-14 * np.abs(b).max())
