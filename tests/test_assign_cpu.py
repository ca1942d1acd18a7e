"""Host assignment engine (include/lpsim_assign.h): time-dependent shortest
paths against brute-force path enumeration, the relative-gap formula, MSA
re-routing, route loading and link-time tables.  Runs on the CPU."""
from __future__ import annotations

import itertools
import math

import numpy as np
import pytest

from netutil import make_net


@pytest.fixture(scope="module")
def A():
    import paper_2406_08496_gb300 as L
    L.build()
    from paper_2406_08496_gb300 import assignment
    return assignment


def _diamond():
    # 0 -> 1 -> 3, 0 -> 2 -> 3, 1 -> 2, plus 3 -> 0 so every node has an out-edge
    edges = [(0, 1, 100.0, 1, 10.0), (1, 3, 100.0, 1, 10.0), (0, 2, 150.0, 1, 10.0), (2, 3, 40.0, 1, 10.0),
             (1, 2, 30.0, 1, 10.0), (3, 0, 50.0, 1, 10.0)]
    net = make_net(4, edges)
    return net, edges


def _cost_ms(seconds):
    """A link time in whole milliseconds (nearest, at least 1 ms)."""
    return max(1, int(math.floor(float(seconds) * 1000.0 + 0.5)))


def _arrival(path, t0, tt, bin_s):
    """Arrival time (s) of a path entered at t0 (s).  A link entered at t
    (ms) in bin b (the last bin beyond the table) is left at the earliest of
    t + c[b] and, for every later bin b', the start of b' + c[b'] (the entry
    may be held back to a later bin); times are whole milliseconds."""
    t = int(math.floor(t0 * 1000.0 + 0.5))
    bin_ms = int(round(bin_s * 1000.0))
    nb = tt.shape[1]
    for e in path:
        b = min(t // bin_ms, nb - 1)
        t = min([t + _cost_ms(tt[e, b])] + [b2 * bin_ms + _cost_ms(tt[e, b2]) for b2 in range(b + 1, nb)])
    return t / 1000.0


def _all_paths(edges, s, d):
    out = []
    adj = {}
    for i, (u, v, *_r) in enumerate(edges):
        adj.setdefault(u, []).append((i, v))

    def rec(u, seen, path):
        if u == d:
            out.append(list(path))
            return
        for i, v in adj.get(u, []):
            if v not in seen:
                rec(v, seen | {v}, path + [i])
    rec(s, {s}, [])
    return out


def test_time_dependent_paths_match_brute_force(A):
    net, edges = _diamond()
    rng = np.random.default_rng(1)
    n_bins, bin_steps, dt = 6, 20, 0.5
    bin_s = bin_steps * dt
    for trial in range(30):
        # FIFO link times: consecutive bins differ by less than a bin width
        base = rng.uniform(2.0, 30.0, (6, 1))
        tt = (base + np.cumsum(rng.uniform(-2.0, 2.0, (6, n_bins)), axis=1)).clip(1.0).astype(np.float32)
        dep = np.array([0, 13, 31, 55, 70], np.uint32)
        dem = {"orig": np.zeros(5, np.uint32), "dest": np.full(5, 3, np.uint32), "depart_step": dep,
               "route_off": np.arange(0, 11, 2, dtype=np.uint64), "route_edges": np.array([0, 1] * 5, np.uint32)}
        a = A.Assignment(net, dem, dt=dt, seed=3)
        period = 10
        tsp = a.shortest_paths(tt, bin_steps, period, n_threads=2)
        a.reroute(1.0, 0)
        routes = a.routes()
        for j in range(5):
            t0 = ((dep[j] // period) + 0.5) * period * dt
            best = min(_arrival(p, t0, tt, bin_s) for p in _all_paths(edges, 0, 3))
            r = routes["route_edges"][int(routes["route_off"][j]):int(routes["route_off"][j + 1])]
            # the route is an earliest-arrival path from the period's middle ...
            assert _arrival(list(r), t0, tt, bin_s) == best
            # ... and its time is counted from the trip's own departure
            tj = float(dep[j]) * dt
            assert abs(tsp[j] - (_arrival(list(r), tj, tt, bin_s) - tj)) < 1e-3


def test_gap_formula(A):
    net, _ = _diamond()
    dem = {"orig": np.zeros(3, np.uint32), "dest": np.full(3, 3, np.uint32), "depart_step": np.array([0, 10, 20], np.uint32),
           "route_off": np.array([0, 2, 4, 6], np.uint64), "route_edges": np.array([0, 1, 0, 1, 0, 1], np.uint32)}
    a = A.Assignment(net, dem, dt=0.5)
    tt = np.full((6, 4), 5.0, np.float32)
    tsp = a.shortest_paths(tt, 100, 100)
    assert np.allclose(tsp, 10.0)  # 0 -> 2 -> 3 or 0 -> 1 -> 3: two links of 5 s
    dep_act = np.array([1, 11, 21], np.uint32)
    arr = np.array([40, 50, 0xFFFFFFFF], np.uint32)  # third trip has not arrived
    rg, used = a.gap(dep_act, arr)
    # experienced 20 s and 20 s against 10 s shortest each: (10 + 10) / 20
    assert used == 2 and abs(rg - 1.0) < 1e-12


def test_reroute_fraction_and_load(A):
    import workloads as W
    net = W.grid_network(5, 5)
    dem = W.route(net, W.uniform_demand(net, 400, 2, t_max_s=600.0))
    a = A.Assignment(net, dem, dt=0.5, seed=7)
    ne = net["n_edges"]
    tt = np.tile((net["edge_len"] / net["edge_vmax"]).astype(np.float32)[:, None], (1, 8))
    tt[::3] *= 3.0  # make some links slow so shortest paths change
    a.shortest_paths(tt, 300, 300)
    assert a.reroute(0.0, 0) == 0
    n1 = a.reroute(0.5, 1)
    n2 = a.reroute(1.0, 2)
    assert 0 < n1 and n1 + n2 > 0
    routes = a.routes()
    # loading: brute-force inflow per (edge, bin)
    inflow = a.load(tt, 300)
    ref = np.zeros((ne, 8), np.int64)
    off = routes["route_off"].astype(np.int64)
    for j in range(len(dem["depart_step"])):
        t = float(dem["depart_step"][j]) * 0.5
        for e in routes["route_edges"][off[j]:off[j + 1]]:
            b = int(math.floor(t / 150.0))
            if 0 <= b < 8:
                ref[e, b] += 1
            t += float(tt[e, min(max(b, 0), 7)])
    assert np.array_equal(inflow, ref)


def test_link_times_and_features(A):
    import workloads as W
    net = W.grid_network(4, 4)
    dem = W.route(net, W.uniform_demand(net, 50, 3))
    a = A.Assignment(net, dem, dt=0.5)
    ne = net["n_edges"]
    s = np.zeros((ne, 4), np.uint32)
    c = np.zeros((ne, 4), np.uint32)
    s[0, 1], c[0, 1] = 300, 3   # 100 steps = 50 s on average
    tt, lr = a.link_times(s, c)
    ff = net["edge_len"] / net["edge_vmax"]
    assert abs(tt[0, 1] - 50.0) < 1e-4 and abs(lr[0, 1] - math.log(50.0 / ff[0])) < 1e-5
    assert np.isnan(lr[1, 1]) and abs(tt[1, 1] - ff[1]) < 1e-4
    y = np.full(ne * 4, math.log(2.0), np.float32)
    tt2 = a.times_from_ratio(y, 4)
    assert np.allclose(tt2, 2.0 * np.repeat(ff[:, None], 4, axis=1), rtol=1e-5)
    X = a.features(np.ones((ne, 4), np.uint32), np.zeros((ne, 4), np.uint32), lr, np.ones((ne, 4), np.uint32))
    assert X.shape == (ne * 4, 11) and np.all(np.isfinite(X))
    assert abs(X[1, 9] - lr[0, 1]) < 1e-6 and X[4 + 1, 9] == 0.0  # unmeasured cells read 0


def test_features_of_listed_cells_equal_all_cells(A):
    """The per-cell feature call gives, bit for bit, the rows of the
    all-cells call for the listed cells, in the listed order; an index past
    the last cell is refused."""
    import workloads as W
    net = W.grid_network(5, 5)
    dem = W.route(net, W.uniform_demand(net, 80, 4))
    a = A.Assignment(net, dem, dt=0.5)
    rng = np.random.default_rng(3)
    ne, nb = net["n_edges"], 12
    inflow = rng.integers(0, 40, (ne, nb)).astype(np.uint32)
    occ = rng.integers(0, 20, (ne, nb)).astype(np.uint32)
    plr = rng.normal(0.0, 0.3, (ne, nb)).astype(np.float32)
    plr[rng.random((ne, nb)) < 0.3] = np.nan
    pin = rng.integers(0, 40, (ne, nb)).astype(np.uint32)
    X = a.features(inflow, occ, plr, pin)
    rows = rng.permutation(ne * nb)[: ne * nb // 3]
    Xr = a.features(inflow, occ, plr, pin, rows=rows)
    assert np.array_equal(X[rows].view(np.uint32), Xr.view(np.uint32))
    assert a.features(inflow, occ, plr, pin, rows=np.zeros(0, np.uint64)).shape == (0, 11)
    with pytest.raises(RuntimeError):
        a.features(inflow, occ, plr, pin, rows=np.array([ne * nb], np.uint64))


def test_worst_first_reroute(A):
    """Per-trip excess from a simulated outcome (gap) and from predicted link
    times (route_excess); worst-first re-routing moves exactly the requested
    share, largest relative excess first, never a trip already on its
    candidate path."""
    import workloads as W
    net = W.grid_network(5, 5)
    dem = W.route(net, W.uniform_demand(net, 300, 4, t_max_s=600.0))
    n = len(dem["depart_step"])
    ff = (net["edge_len"] / net["edge_vmax"]).astype(np.float32)
    tt = np.tile(ff[:, None], (1, 8))
    tt[::3] *= 3.0
    bin_steps = 300
    a = A.Assignment(net, dem, dt=0.5, seed=2)
    tsp = a.shortest_paths(tt, bin_steps, 300)
    a.route_excess(tt, bin_steps)
    # reference: each trip's current route traversed under tt, minus its shortest time
    off = dem["route_off"].astype(np.int64)
    exc = np.empty(n)
    for j in range(n):
        t0 = float(dem["depart_step"][j]) * 0.5
        t = t0
        for e in dem["route_edges"][off[j]:off[j + 1]]:
            t += float(tt[e, min(max(int(math.floor(t / 150.0)), 0), 7)])
        exc[j] = t - t0 - tsp[j]
    before = a.routes()
    moved = a.reroute_worst(0.1)
    after = a.routes()

    def route(r, j):
        return tuple(r["route_edges"][int(r["route_off"][j]):int(r["route_off"][j + 1])])
    changed = [j for j in range(n) if route(before, j) != route(after, j)]
    # the candidates: the same engine state moved wholesale
    b = A.Assignment(net, dem, dt=0.5, seed=2)
    b.shortest_paths(tt, bin_steps, 300)
    b.reroute(1.0, 0)
    cand = b.routes()
    eligible = [j for j in range(n) if exc[j] > 0 and route(cand, j) != route(before, j)]
    rel = exc / np.maximum(1.0, tsp)
    want = min(len(eligible), round(0.1 * n))
    top = sorted(eligible, key=lambda j: (-rel[j], j))[:want]
    assert moved == want > 0
    # same set up to float32 rounding of the excess at the cut
    assert len(set(changed) ^ set(top)) <= 2
    assert all(route(after, j) == route(cand, j) for j in changed)
    # a simulated outcome: the gap call resets the excess from experienced times
    dep_act = dem["depart_step"].astype(np.uint32)
    arr = np.full(n, 0xFFFFFFFF, np.uint32)  # nobody arrived: no excess, nothing moves
    a.gap(dep_act, arr)
    assert a.reroute_worst(0.5) == 0


def _lattice_engine(A, side, n_trips, seed):
    """Trips on a lattice, each on its shortest path under some link times."""
    rng = np.random.default_rng(seed)
    i = np.arange(side * side)
    r, c = np.divmod(i, side)
    src = np.concatenate([i[c < side - 1], i[c > 0], i[r < side - 1], i[r > 0]])
    dst = np.concatenate([i[c < side - 1] + 1, i[c > 0] - 1, i[r < side - 1] + side, i[r > 0] - side])
    net = make_net(side * side, [(int(u), int(v), 100.0, 1, 10.0) for u, v in zip(src, dst)])
    o = rng.integers(0, side * side, 8).repeat(-(-n_trips // 8))[:n_trips]
    d = rng.integers(0, side * side, n_trips)
    dem = {"orig": o.astype(np.uint32), "dest": np.where(d == o, (d + 1) % side ** 2, d).astype(np.uint32),
           "depart_step": rng.integers(0, 4000, n_trips).astype(np.uint32),
           "route_off": np.arange(n_trips + 1, dtype=np.uint64), "route_edges": np.zeros(n_trips, np.uint32)}
    a = A.Assignment(net, dem, seed=seed)
    a.shortest_paths(rng.uniform(5, 30, (len(src), 4)).astype(np.float32), 900, 600)
    a.reroute(1.0, 0)
    return net, dem, a, rng


def _split(routes):
    off = routes["route_off"].astype(np.int64)
    return [routes["route_edges"][off[j]:off[j + 1]].tolist() for j in range(len(off) - 1)]


@pytest.mark.parametrize("n_trips", [1, 7, 500, 20000])
def test_reroutings_of_every_size_leave_the_other_routes(A, n_trips):
    """Small and large re-routings one after another (new routes behind the old
    ones, all in order again when there is no room): exactly the trips counted as
    moved have their candidate path, all others the route they had; the routes read
    back load like those of a new engine."""
    net, dem, a, rng = _lattice_engine(A, 9, n_trips, 3)
    m = net["n_edges"]
    for it, f in enumerate([0.01, 0.02, 0.0, 0.3, 0.05, 0.1, 0.1, 0.1, 1.0, 0.01, 0.6, 0.03]):
        tt = rng.uniform(5, 30, (m, 4)).astype(np.float32)
        before = _split(a.routes())
        b = A.Assignment(net, dict(dem, **{k: v for k, v in a.routes().items() if k != "depart_step"}), seed=9)
        a.shortest_paths(tt, 900, 600)
        b.shortest_paths(tt, 900, 600)
        b.reroute(1.0, 0)
        cand = _split(b.routes())
        if it % 2:
            a.route_excess(tt, 900)
            moved = a.reroute_worst(f)
        else:
            moved = a.reroute(f, it)
        routes = a.routes()
        after = _split(routes)
        differ = [j for j in range(n_trips) if after[j] != before[j]]
        assert len(differ) == moved and all(after[j] == cand[j] for j in differ)
        if f == 1.0 and not it % 2:
            assert after == cand
        c = A.Assignment(net, dict(dem, route_off=routes["route_off"], route_edges=routes["route_edges"]), seed=9)
        assert np.array_equal(a.load(tt, 900), c.load(tt, 900))
        b.close()
        c.close()
    a.close()
