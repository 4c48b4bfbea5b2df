"""The named-barrier hand-over of the encounter kernel's roles (k_bs_ws), modelled on the
CPU: role 0 (R warps) posts evaluation points and takes accelerations, roles 1 and 2 (RM
warps each) take the mutual terms of the even and odd points (above four members the
pairs' terms first, then, in R of the warps and after the stellar terms have arrived, each
member's sum), role 3 (R warps) the stellar term of every point and, two points after a
sequence has ended, its tableau row.  Random interleavings and random accepted
rows over several substeps must never deadlock, no barrier may be met by more warps than
it counts, and every buffer (points, accelerations, stellar terms, raw results, the halt
flag) must hold what its reader expects.  Leaving out a barrier must be caught.
"""
import random

import pytest

LAST = 16   # the last sequence's points


def run(seed, R, RM, nsub=4, leave_out=None):
    rnd = random.Random(seed)
    need = {"P0": 2 * R + RM, "P1": 2 * R + RM, "A0": 3 * R, "A1": 3 * R, "S0": 2 * R, "S1": 2 * R, "row": R,
            "halt": R, "pair0": RM, "pair1": RM}
    count = {b: 0 for b in need}
    gen = {b: 0 for b in need}
    S = {"kacc": -1, "stop": False, "halt": None, "rows": 0}
    pos, sacc, acc, raw, terms = {}, {}, {}, {}, {}     # (buffer, warp of the role) -> tag

    def meet(b, blocking=True):
        if b == leave_out:
            return None
        count[b] += 1
        assert count[b] <= need[b], b
        g = gen[b]
        if count[b] == need[b]:
            count[b] = 0
            gen[b] += 1
        return ("wait", b, g) if blocking else None

    def role0(w):
        for sub in range(nsub):
            accept = S[("accept", sub)]
            pos[0, w], pos[1, w] = (sub, 0), (sub, 1)
            if w == 0:
                S["kacc"], S["stop"] = -1, False
            yield meet("P0", False)
            yield meet("P1", False)
            m = 0
            while True:
                par = m & 1
                yield meet(f"A{par}")
                for q in range(R):      # a lane's acceleration is another warp's
                    assert acc[par, q] == (sub, m)
                pos[par, w] = (sub, m + 2)
                if m >= 2 and par == 0:
                    raw[(m // 2 - 1) & 1, w] = (sub, m // 2 - 1)
                yield meet(f"P{par}", False)
                st = None
                if w == 0:
                    st = S["kacc"] >= 0 or m == LAST
                if RM == 1:
                    stop = st
                else:
                    if w == 0:
                        S["halt"] = (sub, m, st)
                    yield meet("halt")
                    assert S["halt"][:2] == (sub, m)
                    stop = S["halt"][2]
                yield None
                if stop:
                    yield meet(f"A{1 - par}")
                    yield meet(f"A{par}")
                    if w == 0:
                        S["stop"] = True
                    yield meet("P0", False)
                    yield meet("P1", False)
                    break
                m += 1
            yield ("block",)
            assert S["kacc"] == accept
            yield ("block",)

    def role3(w):
        for sub in range(nsub):
            accept = S[("accept", sub)]
            m = 0
            while True:
                par = m & 1
                yield meet(f"P{par}")
                if S["stop"]:
                    yield meet(f"P{1 - par}")
                    break
                for q in range(R):
                    assert pos[par, q] == (sub, m)
                sacc[par, w] = (sub, m)
                if RM > 1:
                    yield meet(f"S{par}", False)
                yield meet(f"A{par}", False)
                if m >= 4 and par == 0:
                    kr = m // 2 - 2
                    for q in range(R):
                        assert raw[kr & 1, q] == (sub, kr)
                    yield None
                    for q in range(R):
                        assert raw[kr & 1, q] == (sub, kr)   # still there when the row is done
                    if kr >= 1:
                        if RM > 1:
                            yield meet("row")
                        if w == 0 and kr == accept and S["kacc"] < 0:
                            S["kacc"] = kr
                m += 1
            yield ("block",)
            yield ("block",)

    def mutual(w, par):
        for sub in range(nsub):
            m = par
            while True:
                yield meet(f"P{par}")
                if S["stop"]:
                    break
                for q in range(R):
                    assert pos[par, q] == (sub, m)
                if RM > 1:
                    terms[par, w] = (sub, m)
                    yield meet(f"pair{par}")
                if w < R:
                    if RM > 1:
                        yield meet(f"S{par}")
                        for q in range(R):
                            assert sacc[par, q] == (sub, m)
                        for q in range(RM):
                            assert terms[par, q] == (sub, m)
                        yield None
                        for q in range(RM):
                            assert terms[par, q] == (sub, m)
                    acc[par, w] = (sub, m)
                    yield meet(f"A{par}", False)
                m += 2
            yield ("block",)
            yield ("block",)

    for sub in range(nsub):
        S["accept", sub] = rnd.choice([-1, 1, 2, 3, 4, 5, 6, 7])
    warps = {}
    for w in range(R):
        warps["state", w] = role0(w)
        warps["star", w] = role3(w)
    for w in range(RM):
        warps["even", w] = mutual(w, 0)
        warps["odd", w] = mutual(w, 1)
    pending = {k: None for k in warps}
    done, blocked, nblock, steps = set(), set(), 0, 0
    while len(done) < len(warps):
        steps += 1
        assert steps < 200000, "livelock"
        ready = []
        for k, p in pending.items():
            if k in done:
                continue
            if p is None or (p[0] == "wait" and gen[p[1]] > p[2]) or (p[0] == "block" and nblock > p[1]):
                ready.append(k)
        assert ready, ("deadlock", pending)
        k = rnd.choice(ready)
        try:
            r = next(warps[k])
        except StopIteration:
            done.add(k)
            continue
        if r is not None and r[0] == "block":
            blocked.add(k)
            r = ("block", nblock)
            if len(blocked) == len(warps):
                blocked.clear()
                nblock += 1
        pending[k] = r
    assert all(v == 0 for v in count.values()), count


@pytest.mark.parametrize("R,RM", [(1, 1), (2, 6), (3, 5), (4, 4)])
def test_roles_hand_over(R, RM):
    for seed in range(150):
        run(seed, R, RM)


@pytest.mark.parametrize("barrier", ["S0", "S1", "halt", "pair0", "pair1"])
def test_a_missing_barrier_is_caught(barrier):
    with pytest.raises((AssertionError, KeyError, TypeError)):
        for seed in range(60):
            run(seed, 2, 6, leave_out=barrier)
