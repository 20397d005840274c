"""The colouring by arrivals, modelled on the CPU: whoever colours a contact
carries the colour masks of its two lists on to the contacts that follow it
there, the first of two arrivals at a contact leaves its mask, the last one
takes it up and the contact is coloured next.  Whatever the order in which
the contacts at hand are taken, the colours are those of the sequential
first-fit greedy colouring in decreasing priority.  (The GPU's own colours are
compared with the same greedy colouring in tests/test_gpu_colour.py.)"""
import random

import pytest


def _greedy(ends, prio):
    used, col = {}, {}
    for c in sorted(range(len(ends)), key=lambda c: (-prio[c], c)):
        m = 0
        for x in ends[c]:
            m |= used.get(x, 0)
        bit = ~m & (m + 1)
        col[c] = bit.bit_length() - 1
        for x in ends[c]:
            used[x] = used.get(x, 0) | bit
    return col


def _arrivals(ends, prio, rng):
    lists = {}
    for c in sorted(range(len(ends)), key=lambda c: (-prio[c], c)):
        for x in ends[c]:
            lists.setdefault(x, []).append(c)
    succ = {(x, c): l[k + 1] for x, l in lists.items() for k, c in enumerate(l[:-1])}
    preds = {c: sum(lists[x][0] != c for x in ends[c]) for c in range(len(ends))}
    meet, col = {}, {}
    queue = [(c, {}) for c in range(len(ends)) if preds[c] == 0]
    while queue:
        c, masks = queue.pop(rng.randrange(len(queue)))
        m = 0
        for x in ends[c]:
            m |= masks.get(x, 0)
        bit = ~m & (m + 1)
        assert c not in col
        col[c] = bit.bit_length() - 1
        for x in ends[c]:
            e = succ.get((x, c))
            if e is None:
                continue
            brought = {x: masks.get(x, 0) | bit}
            if preds[e] == 1:
                queue.append((e, brought))
            elif e in meet:
                queue.append((e, {**meet.pop(e), **brought}))
            else:
                meet[e] = brought
    assert not meet
    return col


@pytest.mark.parametrize("n,m,seed", [(2, 1, 0), (5, 9, 1), (40, 120, 2), (200, 1000, 3), (30, 200, 4), (500, 600, 5)])
def test_any_order_of_arrivals_gives_the_greedy_colours(n, m, seed):
    rng = random.Random(seed)
    ends = set()
    while len(ends) < min(m, n * (n - 1) // 2 + n):
        a, b = rng.randrange(n), rng.randrange(n)
        ends.add((min(a, b), max(a, b)) if a != b else (a,))   # one end: a wall or a fixed body
    ends = sorted(ends)
    prio = [rng.getrandbits(8) for _ in ends]                 # ties among them
    want = _greedy(ends, prio)
    for _ in range(5):
        assert _arrivals(ends, prio, rng) == want
