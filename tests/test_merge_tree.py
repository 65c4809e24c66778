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


def insert_halving(T, age, s, u, v, far=0):
    """insert_younger whose climbs, after `far` steps, replace a word's root by
    the next one on its path when that is connected below the word's key."""
    steps = 0
    while u != v:
        if age[u] < age[v]:
            u, v = v, u
        yield
        w = T[u]
        steps += 1
        while w[0] > s:
            yield
            if T[u] == w:
                T[u] = (s, v)
                break
            w = T[u]
        else:
            x = w
            if steps > far:
                yield
                x = T[w[1]]
                if x[0] >= s:
                    x = w
                elif x[0] < w[0]:
                    yield
                    if T[u] == w:
                        T[u] = (w[0], x[1])
            u = x[1]
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


def _drive(insert, n, age, edges, rng, width):
    T, todo, live = [(INF, k) for k in range(n)], list(edges), []
    rng.shuffle(todo)
    while todo or live:
        while todo and len(live) < width:
            live.append(insert(T, age, *todo.pop()))
        k = rng.randrange(len(live))
        try:
            next(live[k])
        except StopIteration:
            live.pop(k)
    return T


@pytest.mark.parametrize("width", [1, 2, 5, 64])
@pytest.mark.parametrize("kind", ["random", "slope", "climb", "rungs"])
@pytest.mark.parametrize("far", [0, 3])
def test_any_schedule_with_shortened_paths(far, kind, width):
    rng = random.Random(f"{kind}{width}{far}")
    for trial in range(60):
        n = rng.randint(2, 40)
        age = sorted(rng.sample(range(1000), n))
        if kind == "random":
            rng.shuffle(age)
            ends = [(rng.randrange(n), rng.randrange(n)) for _ in range(rng.randint(0, 4 * n))]
            level = rng.sample(range(10000), len(ends))
        else:
            ends = [(k, k + 1) for k in range(n - 1)]
            level = sorted(rng.sample(range(10000), n - 1), reverse=kind == "climb")
            if kind == "rungs":  # two slopes side by side, and connections between far parts above both
                more = [(rng.randrange(n), rng.randrange(n)) for _ in range(3 * n)]
                ends, level = ends + more, level + rng.sample(range(10000, 20000), len(more))
        edges = [(s, u, v) for s, (u, v) in zip(level, ends)]
        T = _drive(lambda *a: insert_halving(*a, far=far), n, age, edges, rng, width)
        assert [t[0] for t in T] == sequential(n, age, edges)
        assert all(t[0] == INF or age[t[1]] < age[k] for k, t in enumerate(T))


@pytest.mark.gpu
@pytest.mark.parametrize("shape", [(1024, 8192), (8192, 1024), (64, 64, 512)])
def test_slopes_take_short_climbs(shape):
    """Noise on a ramp: the mean climb is no longer than the levels of a balanced
    tree (it was the distance to where the two paths meet: 54, 53 and 49 steps),
    and the pairs are those of the sorted union-find."""
    import ctypes
    import math

    torch = pytest.importorskip("torch")
    import paper_2606_04801_gb300 as cp

    lib = cp.load()
    g = torch.Generator(device="cuda").manual_seed(3)
    ax = max(range(len(shape)), key=lambda k: shape[k])
    slope = torch.arange(shape[ax], device="cuda", dtype=torch.float32).div(16).view([-1 if k == ax else 1 for k in range(len(shape))])
    x = (slope + torch.rand(shape, generator=g, device="cuda")).contiguous()
    dims = (ctypes.c_int64 * len(shape))(*shape)
    ws_bytes = lib.cubical_persistence_workspace_size(len(shape), dims, x.numel())
    ws = torch.empty(ws_bytes, dtype=torch.uint8, device="cuda")
    out = torch.empty((x.numel(), 8), dtype=torch.int32, device="cuda")
    cnt = ctypes.c_int64(0)
    fn = lib.cubical_persistence_2d if len(shape) == 2 else lib.cubical_persistence_3d
    p = lambda t: ctypes.c_void_p(t.data_ptr())  # noqa: E731
    rc = fn(p(x), dims, p(out), x.numel(), ctypes.byref(cnt), None, p(ws), ws_bytes, x.numel(), None)
    assert rc == 0
    act, us, hops = (ctypes.c_uint32 * 48)(), (ctypes.c_double * 48)(), (ctypes.c_uint64 * 48)()
    n = []
    for dual in (0, 1):
        assert lib.cubical_persistence_uf_trace2(p(ws), dual, act, us, None, hops, 48, None) == 2
        n.append(act[0])
        if dual == 0:
            steps = hops[1]
    assert lib.cp_set_tuning(7, 1) == 0
    try:
        want = cp.persistence(x).raw
    finally:
        assert lib.cp_set_tuning(7, 0) == 0
    assert torch.equal(out[: cnt.value], want)
    mean = steps / sum(n)
    assert mean < math.log2(sum(n)), mean
