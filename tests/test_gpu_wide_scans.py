"""The bucket and group scans of more than 32768 counts (a block for every 4096), at sizes
around that line and at a ragged last block: groups, mergers and states of many systems
together against the same systems one at a time, whose scans are the one-block ones.

Each system's arithmetic does not depend on the others beside it but for the kick's tiles, so the
FP64 form agrees to rounding; the counts are whole numbers.
"""
import numpy as np
import pytest

import opal_ic as ic

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sizes", [[300] * 64, [300] * 65, [40] * 300, [5000, 70, 33000], [131000, 1, 900]])
def test_many_systems_together_as_one_at_a_time(sizes):
    from paper_2601_19654_gb300 import opal
    systems = [ic.tiny(100 + k, n) if n < 2000 else ic.equal_mass_disk(k, n) for k, n in enumerate(sizes)]
    with opal.Simulation.ensemble(systems, precision=0, dt=0.02) as sim:
        sim.step(1)
        all_stats = sim.stats()
        states = [sim.state(k) for k in range(len(sizes))]
    total = dict.fromkeys(("n_pairs", "n_groups", "n_candidates"), 0)
    check = range(len(sizes)) if len(sizes) <= 70 else range(0, len(sizes), 7)
    for k, s in enumerate(systems):
        if len(sizes) > 70 and k % 7:
            continue
        with opal.Simulation.from_system(s, precision=0, dt=0.02) as one:
            one.step(1)
            st = one.state()
            for key in total:
                total[key] += one.stats()[key]
        assert st["ids"].tolist() == states[k]["ids"].tolist()
        np.testing.assert_allclose(states[k]["x"], st["x"], rtol=0, atol=1e-9)
    if len(sizes) <= 70:
        assert all(all_stats[key] == total[key] for key in total), (all_stats, total)
    assert len(list(check)) > 0


# Slots of a system are padded to 128: 85 systems of 300 bodies have 32640 slots, 86 have 33024 (the group
# scan's line), 256 of 500 have 32768 buckets, 257 have 32896 (the bucket scan's).  The references are
# small systems one at a time, which take neither scan.
@pytest.mark.parametrize("size,count", [(300, 85), (300, 86), (500, 256), (500, 257)])
def test_counts_at_the_line_as_one_at_a_time(size, count):
    from paper_2601_19654_gb300 import opal
    systems = [ic.tiny(2000 + k, size) for k in range(count)]
    keys = ("n_pairs", "n_groups", "n_candidates", "n_mergers")
    with opal.Simulation.ensemble(systems, precision=0, dt=0.02) as sim:
        sim.step(1)
        together = sim.stats()
        states = [sim.state(k) for k in range(count)]
    alone = dict.fromkeys(keys, 0)
    for s, st in zip(systems, states):
        with opal.Simulation.from_system(s, precision=0, dt=0.02) as one:
            one.step(1)
            stats, ref = one.stats(), one.state()
        for key in keys:
            alone[key] += stats[key]
        assert st["ids"].tolist() == ref["ids"].tolist()
        np.testing.assert_allclose(st["x"], ref["x"], rtol=0, atol=1e-9)
    assert alone["n_groups"] > count
    assert {key: together[key] for key in keys} == alone
