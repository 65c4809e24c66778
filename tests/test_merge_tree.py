"""The merge tree of the union-finds (cp_tree.cu), restated step by step.

Survivors go in one at a time or interleaved at every read and swap, in any
order; the level at which each root stops being the oldest of its class must
be the sequential elder-rule union-find's, whatever the schedule.
"""
import random

import pytest

INF = float("inf")


def insert(T, age, s, u, v):
    """One survivor's thread; yields before every read or swap of a word."""
    while True:
        yield
        wu = T[u]
        yield
        wv = T[v]
        while wu[0] < s or wv[0] < s:
            if wu[0] < s:
                u = wu[1]
                yield
                wu = T[u]
            if wv[0] < s:
                v = wv[1]
                yield
                wv = T[v]
        if u == v:
            return
        if age[u] < age[v]:
            u, v, wu = v, u, wv
        yield
        if T[u] != wu:
            continue
        T[u] = (s, v)
        if wu[0] == INF:
            return
        s, u, v = wu[0], v, wu[1]


def insert_younger(T, age, s, u, v):
    """The same with only the younger end's word read (cp_tree.cu)."""
    while u != v:
        if age[u] < age[v]:
            u, v = v, u
        yield
        w = T[u]
        while w[0] > s:
            yield
            if T[u] == w:
                T[u] = (s, v)
                break
            w = T[u]
        else:
            u = w[1]
            continue
        if w[0] == INF:
            return
        s, u, v = w[0], v, w[1]


def sequential(n, age, edges):
    par, death = list(range(n)), [INF] * n

    def find(a):
        while par[a] != a:
            a = par[a]
        return a

    for s, u, v in sorted(edges):
        u, v = find(u), find(v)
        if u == v:
            continue
        if age[u] < age[v]:
            u, v = v, u
        par[u] = v
        death[u] = s
    return death


@pytest.mark.parametrize("width", [1, 2, 3, 8, 64])
@pytest.mark.parametrize("kind", ["random", "path", "staircase", "star"])
@pytest.mark.parametrize("insert", [insert, insert_younger])
def test_any_schedule_gives_the_elder_rule(insert, kind, width):
    rng = random.Random(f"{kind}{width}")
    for trial in range(60):
        n = rng.randint(1, 24)
        age = rng.sample(range(1000), n)
        if kind == "random":
            ends = [(rng.randrange(n), rng.randrange(n)) for _ in range(rng.randint(0, 4 * n))]
        elif kind == "star":
            ends = [(0, k) for k in range(1, n)] * 2
        else:
            ends = [(k, k + 1) for k in range(n - 1)]
        level = rng.sample(range(10000), len(ends))
        if kind == "staircase":  # nested classes: levels and ages both rise along the path
            age, level = sorted(age), sorted(level, reverse=trial % 2 == 0)
        edges = [(s, u, v) for s, (u, v) in zip(level, ends)]
        T = [(INF, k) for k in range(n)]
        todo = list(edges)
        rng.shuffle(todo)
        live = []
        while todo or live:
            while todo and len(live) < width:
                live.append(insert(T, age, *todo.pop()))
            k = rng.randrange(len(live))
            try:
                next(live[k])
            except StopIteration:
                live.pop(k)
        assert [t[0] for t in T] == sequential(n, age, edges)
        assert all(t[0] == INF or age[t[1]] < age[k] for k, t in enumerate(T))
