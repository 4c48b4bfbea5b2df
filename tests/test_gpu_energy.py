"""The energy's pair sum at the edges of its tiles and of its float-pair form.

The energy diagnostics sum m_i m_j / r_ij over pairs of 128-body tiles, in plain
FP64 below 512 bodies and, tile by tile, where coordinates or masses leave the range
of the float-pair form, in float pairs (hi + lo) otherwise.  Here the star is light
and the bodies are at rest, so that the pair sum is all but the whole energy, which is
compared with the sum in extended precision.

Tolerance: the FP64 sums round at most about 16 times a term along their fixed-order
trees (2^-53 each), and a float-pair term is right to 2^-45, independently from pair
to pair: 2^-45 / sqrt(pairs) of the sum, below 2^-53 from 512 bodies (130816 pairs)
on.  Together under 32 x 2^-53 = 2^-48 of the sum.
"""
import numpy as np
import pytest

import opal_ic as ic

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _system(kind, n):
    s = ic.equal_mass_disk(n, n)
    m, x = s.m.copy(), s.x.copy()
    u = ic.uniform(n, 77, np.arange(n))
    m *= 0.1 + u                       # unequal masses
    if kind == "small_bodies":
        m[n // 2:] = 0.0
    if kind == "cgs":                  # cm and g: out of the float form's range
        x *= ic.AU_CM
        m *= ic.MSUN_G
    if kind == "one_far":              # one body whose units no float pair holds
        x[-1] *= 1e12
    if kind == "close":                # pairs far closer than the float split resolves
        k = n // 2
        x[k:2 * k] = x[:k] + 1e-9 * (u[:k, None] - 0.5)
    return m, x


def _pair_sum(m, x):
    ml, xl = m.astype(np.longdouble), x.astype(np.longdouble)
    total = np.longdouble(0)
    for i in range(len(m) - 1):
        d = xl[i + 1:] - xl[i]
        total += ml[i] * (ml[i + 1:] / np.sqrt((d * d).sum(1))).sum()
    return float(total)


@pytest.mark.parametrize("kind", ["disk", "small_bodies", "cgs", "one_far", "close"])
@pytest.mark.parametrize("n", [2, 33, 129, 511, 512, 641, 1500])
def test_pair_sum_matches_extended_precision(kind, n):
    from paper_2601_19654_gb300 import opal
    m, x = _system(kind, n)
    M0 = 1e-40 * m.sum()
    want = _pair_sum(m, x) + M0 * float((m / np.linalg.norm(x, axis=1)).sum())   # and the light star's share
    t = [torch.as_tensor(a, device="cuda") for a in (m, x, np.zeros_like(x))]
    out = torch.full((7,), float("nan"), dtype=torch.float64, device="cuda")
    st = torch.cuda.current_stream()
    opal.energy_momentum_noalloc(n, 1.0, M0, *(a.data_ptr() for a in t), out.data_ptr(), st.cuda_stream)
    st.synchronize()
    assert abs(-float(out[0]) - want) <= 2.0 ** -48 * want
    # the same sum of a simulation's bodies (small bodies behind the big ones), one system of two
    first = ic.tiny(3, 20)
    with opal.Simulation(np.concatenate([first.m * m.max() / first.m.max(), m]), np.concatenate([first.x, x]),
                         np.zeros((20 + n, 3)), np.zeros(20 + n), n_per_sys=[20, n], M0=M0) as sim:
        E = sim.energy(1)[0]
    assert abs(-E - want) <= 2.0 ** -48 * want
