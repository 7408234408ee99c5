"""The controller's colouring window, modelled on the host.

A window runs up to 31 quiet sweeps at once (see test_colour_pass_model.py for
why a run of quiet sweeps is a first-fit edge colouring in position order).
This test replays its procedure step by step -- lists of the next edges that
still have a free colour below the bound, groups of 32, rounds in which every
edge without a pending earlier neighbour takes its lowest free colour and one
busy agent's edges take its free colours in order, the bound falling at
applicable edges and at edges that come back, and the bound halved after a
budget of coloured edges -- on random hub-heavy edge lists, and checks it
against sweeps simulated one by one."""
import random

import pytest

from test_colour_pass_model import random_case, sweeps_one_by_one


def window(live, refresh, cand, limit=31, budget=1 << 30, busy_at=4):
    """(F, per-sweep counts, edges left, an event follows)."""
    mask, colour = {}, {}
    cap = (1 << min(limit, 31)) - 1
    below = None
    order = sorted(live)
    cursor, next_budget = 0, budget

    def free_of(p):
        u, v, _ = live[p]
        return ~(mask.get(u, 0) | mask.get(v, 0)) & cap

    while cap and cursor < len(order):
        listed = []
        while cursor < len(order) and len(listed) < cand:
            if free_of(order[cursor]):
                listed.append(order[cursor])
            cursor += 1
        for g in range(0, len(listed), 32):
            if not cap:
                break
            group = listed[g:g + 32]
            ends = [set(live[p][:2]) for p in group]
            conf = [{j for j in range(i) if ends[j] & ends[i]} for i in range(len(group))]
            busy = any(len(c) >= busy_at for c in conf)
            mine = [0] * len(group)
            pend = [i for i, p in enumerate(group) if free_of(p)]
            while pend:
                low = {i: free_of(group[i]) & -free_of(group[i]) for i in pend if not conf[i] & set(pend)}
                if busy:
                    u, v, _ = live[group[pend[0]]]
                    at_u = [i for i in pend if u in ends[i]]
                    at_v = [i for i in pend if v in ends[i]]
                    hub, at_h = (u, at_u) if len(at_u) >= len(at_v) else (v, at_v)
                    free = ~mask.get(hub, 0) & cap
                    bits = [b for b in range(31) if free >> b & 1]
                    for r, i in enumerate(at_h):
                        a, b, _ = live[group[i]]
                        other = b if a == hub else a
                        if mask.get(other, 0) & free or conf[i] & (set(pend) - set(at_h)):
                            break
                        low[i] = 1 << bits[r] if r < len(bits) else 0
                for i, c in low.items():
                    if c and live[group[i]][2]:
                        below = c - 1 if below is None else min(below, c - 1)
                bound = cap
                for i, c in low.items():
                    if c and live[group[i]][2]:
                        bound &= c - 1
                    elif c and refresh[group[i]] is not None:
                        bound &= (c << 1) - 1
                cap = bound
                for i, c in low.items():
                    if c & cap and not live[group[i]][2]:
                        mine[i] = c
                        for a in ends[i]:
                            mask[a] = mask.get(a, 0) | c
                pend = [i for i, p in enumerate(group) if not mine[i] and free_of(p)]
            for i, c in enumerate(mine):
                if c:
                    colour[group[i]] = c.bit_length() - 1
            if len(colour) >= next_budget:
                next_budget += budget
                cap &= cap >> ((bin(cap).count("1") + 1) // 2)
    bound = bin(cap).count("1")
    hist = [sum(1 for c in colour.values() if c == k) for k in range(bound)]
    F = sum(1 for h in hist if h)
    out = dict(live)
    for p, c in colour.items():
        if c < F:
            if refresh[p] is None:
                del out[p]
            else:
                out[p] = (refresh[p][0], refresh[p][1], True)
    return F, hist[:F], out, below == cap and bound == F


@pytest.mark.parametrize("seed", range(60))
@pytest.mark.parametrize("cand,budget", [(128, 1 << 30), (64, 40), (32, 377)])
def test_window_equals_quiet_sweeps(seed, cand, budget):
    rng = random.Random(seed)
    live, refresh = random_case(rng)
    for _ in range(200):
        f, counts, after, event = window(live, refresh, cand, limit=rng.choice([31, 31, 5]), budget=budget)
        ref_counts, ref_live = sweeps_one_by_one(live, refresh, f)
        assert counts == ref_counts and len(ref_counts) == f
        if f:
            assert after == ref_live
        if event:  # the next sweep commits
            assert sweeps_one_by_one(after, refresh, 1)[0] == [] and after
        if f == 0 or not after:
            break
        live = after
        refresh = {p: (refresh[p] if not live[p][2] else None) for p in live}
