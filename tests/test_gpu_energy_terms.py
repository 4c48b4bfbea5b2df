"""The energy's pair sum where few terms carry it, or where its separations cancel: one body with
most of the sum in front of a disk, two with nearly all of it, a compact clump far from the
star, a distant straggler beside a disk, and massless bodies wherever they are.

Against the sum in extended precision, to 2^-50 of it.  A term's 1 / r is right to 3 x 2^-53
and is added by one FP64 FMA.  A thread adds at most 128 terms in a row, whose roundings (2^-53 of the
running sum at most, 0.3 x 2^-53 rms, the sum growing by equal terms) come to about 0.3 x sqrt(128 / 3) = 2 x
2^-53 of the thread's sum, independent from thread to thread.  With a term's own error
where one pair is nearly the whole sum (3), the trees (7 + 8 levels of 0.3 rms: about 1) and the rounding of the
reference (1/2) that is below 8 x 2^-53.  (Runs of 128 terms in two floats were off by 2^-47.5 rms of one body's sum.)
"""
import numpy as np
import pytest

import opal_ic as ic

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _system(kind, n):
    s = ic.equal_mass_disk(n, n)
    m, x = s.m.copy(), s.x.copy()
    u = np.stack([ic.uniform(n, 78 + k, np.arange(n)) for k in range(3)], 1)
    if kind == "heavy":                # n / 6000 of the others' mass: most of the sum
        m[n // 3] = max(1.0, n / 6000) * m.sum()
    if kind == "pair":                 # one pair is all but the whole sum
        m[1] = m[n - 2] = 1e6 * m.sum()
    if kind == "clump":                # within 0.01 to 0.05 of |x|
        x = np.array([30.0, 3.0, 0.3]) + 0.9 * (u - 0.5)
    if kind == "straggler":            # its tiles' unit of length is 1000 times the others'
        x[n // 2] *= 1e5 / np.linalg.norm(x[n // 2])
    if kind == "massless":
        m[::3] = 0.0
        x[0], x[3], x[6] = 0.0, [1e300, 0.0, 0.0], x[7]
    if kind == "kilometres":
        x *= 1.495978707e8
    return m, x


def _pair_sum(m, x):
    i = np.nonzero(m)[0]
    ml, xl = m[i].astype(np.longdouble), x[i].astype(np.longdouble)
    total = np.longdouble(0)
    for k in range(len(ml) - 1):
        d = xl[k + 1:] - xl[k]
        total += ml[k] * (ml[k + 1:] / np.sqrt((d * d).sum(1))).sum()
    return float(total)


@pytest.mark.parametrize("kind", ["heavy", "pair", "clump", "straggler", "massless", "kilometres"])
@pytest.mark.parametrize("n", [40, 513, 1500, 4224])
def test_pair_sum_of_unequal_terms(kind, n):
    from paper_2601_19654_gb300 import opal
    m, x = _system(kind, n)
    M0 = 1e-40 * m.sum()
    want = _pair_sum(m, x)             # (the star's share is 1e-40 of it)
    t = [torch.as_tensor(a, device="cuda") for a in (m, x, np.zeros_like(x))]
    out = torch.full((7,), float("nan"), dtype=torch.float64, device="cuda")
    st = torch.cuda.current_stream()
    opal.energy_momentum_noalloc(n, 1.0, M0, *(a.data_ptr() for a in t), out.data_ptr(), st.cuda_stream)
    st.synchronize()
    assert abs(-float(out[0]) - want) <= 2.0 ** -50 * want
    if kind == "massless":
        return                         # (a simulation has its massless bodies last)
    with opal.Simulation(m, x, np.zeros((n, 3)), np.zeros(n), M0=M0) as sim:
        E = sim.energy()[0]
    assert abs(-E - want) <= 2.0 ** -50 * want


# 2^-51: one body holds two thirds of the sum in 64 runs of 128 terms of one thread, whose roundings come
# to 2 / sqrt(64) x 2^-53; with the trees and the last operations about 0.7 x 2^-53 rms.  The reference adds FP64
# terms without rounding (their own errors average to 0.01 x 2^-53).
@pytest.mark.parametrize("seed", [0, 1, 2])
def test_one_body_as_heavy_as_all_others(seed):
    import math

    from paper_2601_19654_gb300 import opal
    n = 8192
    s = ic.equal_mass_disk(seed + 10 * n, n)
    m, x = s.m.copy(), s.x
    m[0] = m.sum()
    rows = []
    for k in range(n - 1):
        d = x[k + 1:] - x[k]
        rows.append(m[k] * math.fsum(m[k + 1:] / np.sqrt((d * d).sum(1))))
    want = math.fsum(rows)
    t = [torch.as_tensor(np.ascontiguousarray(a), device="cuda") for a in (m, x, np.zeros_like(x))]
    out = torch.full((7,), float("nan"), dtype=torch.float64, device="cuda")
    st = torch.cuda.current_stream()
    opal.energy_momentum_noalloc(n, 1.0, 1e-40 * m.sum(), *(a.data_ptr() for a in t), out.data_ptr(), st.cuda_stream)
    st.synchronize()
    assert abs(-float(out[0]) - want) <= 2.0 ** -51 * want
