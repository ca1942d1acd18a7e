"""The assignment loop on the GPU: plain MSA and surrogate-assisted MSA on a
small regional case; every gap is measured by a full simulation; on the
regional day the trained surrogate predicts link times better than the
method without it (the last simulation's own times)."""
from __future__ import annotations

import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import paper_2406_08496_gb300 as L
    L.build()
    L.load_library()
    L.use_torch_allocator()


@pytest.fixture(scope="module")
def case():
    return W.assignment_case(scale="tiny")


def _tables(net, n_bins, seed, spread=0.8):
    """Link-time tables around free flow, each (edge, bin) scaled by its own
    random factor -- times fall as well as rise between bins, so the FIFO
    rule (holding an entry back to a later bin) is exercised."""
    rng = np.random.default_rng(seed)
    ff = (net["edge_len"] / net["edge_vmax"]).astype(np.float64)[:, None]
    return (ff * np.exp(rng.uniform(0.0, spread, (net["n_edges"], n_bins)))).astype(np.float32)


def _paths(A, search, tt, bin_steps, period_steps):
    tsp = search(tt, bin_steps, period_steps)
    A.reroute(1.0, 0)  # every trip takes its candidate: the routes are the paths
    return tsp, A.routes()


@pytest.mark.parametrize("scale,period_steps,seed", [("tiny", 3600, 1), ("tiny", 600, 2), ("tiny", 36000, 3),
                                                     ("small", 3600, 4)])
def test_gpu_paths_equal_host_paths(scale, period_steps, seed):
    """The GPU search (one warp per tree, label-correcting rounds on packed
    (arrival, edge) labels) returns the host Dijkstra's routes and times bit
    for bit: the earliest arrival, ties to the lower entering edge id."""
    from paper_2406_08496_gb300.assignment import Assignment
    net, dem = W.assignment_case(scale=scale)
    tt = _tables(net, 96, seed)
    host = Assignment(net, dem, seed=seed)
    gpu = Assignment(net, dem, seed=seed)
    th, rh = _paths(host, host.shortest_paths, tt, 1800, period_steps)
    tg, rg = _paths(gpu, gpu.shortest_paths_gpu, tt, 1800, period_steps)
    assert np.array_equal(th.view(np.uint32), tg.view(np.uint32))
    assert np.array_equal(rh["route_off"], rg["route_off"])
    assert np.array_equal(rh["route_edges"], rg["route_edges"])
    # a second call on the same engine reuses its device state
    tt2 = _tables(net, 96, seed + 10)
    th2 = host.shortest_paths(tt2, 1800, period_steps)
    tg2 = gpu.shortest_paths_gpu(tt2, 1800, period_steps)
    assert np.array_equal(th2.view(np.uint32), tg2.view(np.uint32))
    host.close()
    gpu.close()


@pytest.mark.parametrize("scale", ["tiny", "small"])
def test_gpu_load_equals_host_load(scale):
    """Inflow per (edge, bin) of the current routes walked on the GPU equals
    the host walk, count for count, before and after a re-routing."""
    from paper_2406_08496_gb300.assignment import Assignment
    net, dem = W.assignment_case(scale=scale)
    tt = _tables(net, 96, 7)
    A = Assignment(net, dem, seed=2)
    assert np.array_equal(A.load(tt, 1800), A.load_gpu(tt, 1800))
    A.shortest_paths_gpu(tt, 1800, 3600)
    A.reroute(0.3, 1)
    tt2 = _tables(net, 96, 8)
    ref = A.load(tt2, 1800)
    assert ref.sum() > 0
    assert np.array_equal(ref, A.load_gpu(tt2, 1800))
    A.close()


def _lattice(side):
    i = np.arange(side * side)
    r, c = np.divmod(i, side)
    src = np.concatenate([i[c < side - 1], i[c > 0], i[r < side - 1], i[r > 0]])
    dst = np.concatenate([i[c < side - 1] + 1, i[c > 0] - 1, i[r < side - 1] + side, i[r > 0] - side])
    return side * side, src, dst


def _odd_network(kind):
    """{nodes, edge tails, edge heads, origins and destinations of trips}"""
    rng = np.random.default_rng(5)
    if kind == "hub":  # 3,000 nodes reached in one round
        n = 3000
        src = np.concatenate([np.zeros(n, int), np.arange(1, n + 1)])
        dst = np.concatenate([np.arange(1, n + 1), np.full(n, n + 1)])
        return n + 2, src, dst, np.zeros(40, int), np.concatenate([np.full(20, n + 1), rng.integers(1, n + 1, 20)])
    if kind == "line":  # paths of up to 1,499 edges
        n = 1500
        return n, np.arange(n - 1), np.arange(1, n), np.zeros(40, int), rng.integers(1, n, 40)
    n, src, dst = _lattice(int(kind))
    o = rng.integers(0, n, 12).repeat(8)
    d = rng.integers(0, n, len(o))
    return n, src, dst, o, np.where(d == o, (d + 1) % n, d)


@pytest.mark.parametrize("kind", ["2", "5", "hub", "line", "90", "91", "236", "237"])
@pytest.mark.parametrize("n_bins,shuffled", [(1, True), (33, False), (96, True)])
def test_gpu_paths_on_odd_networks(kind, n_bins, shuffled):
    """Where the search can go wrong: a tree of a few nodes, more waiting nodes
    than the ring of ids holds, paths longer than the walk's scratch, networks on
    both sides of each choice of block (90 x 90 and 91 x 91 nodes) and of the
    largest whose labels fit in shared memory (236 x 236 do, 237 x 237 do
    not), edge ids in no order, and link times of one to three seconds, so that
    many paths tie: routes and times equal the host's bit for bit."""
    from paper_2406_08496_gb300.assignment import Assignment
    n, src, dst, o, d = _odd_network(kind)
    rng = np.random.default_rng(6)
    if shuffled:
        p = rng.permutation(len(src))
        src, dst = src[p], dst[p]
    m = len(src)
    net = {"n_nodes": n, "n_edges": m, "edge_src": src.astype(np.uint32), "edge_dst": dst.astype(np.uint32),
           "edge_len": np.full(m, 100.0, np.float32), "edge_lanes": np.ones(m, np.uint8),
           "edge_vmax": np.full(m, 10.0, np.float32)}
    dem = {"orig": o.astype(np.uint32), "dest": d.astype(np.uint32),
           "depart_step": rng.integers(0, 4000, len(o)).astype(np.uint32),
           "route_off": np.arange(len(o) + 1, dtype=np.uint64), "route_edges": np.zeros(len(o), np.uint32)}
    tt = rng.integers(1, 4, (m, n_bins)).astype(np.float32)
    host, gpu = Assignment(net, dem, seed=1), Assignment(net, dem, seed=1)
    for period in (600, 7):
        th, rh = _paths(host, host.shortest_paths, tt, 60, period)
        tg, rg = _paths(gpu, gpu.shortest_paths_gpu, tt, 60, period)
        assert np.array_equal(th.view(np.uint32), tg.view(np.uint32))
        assert np.array_equal(rh["route_off"], rg["route_off"])
        assert np.array_equal(rh["route_edges"], rg["route_edges"])
        assert np.array_equal(host.load(tt, 60), gpu.load_gpu(tt, 60))
    # times that round to less than a millisecond, to a half, and past 2^31 ms
    odd = rng.choice(np.array([0.0, -3.0, 1e-4, 0.0005, 0.0025, 1.5, 2147483.5, 3e6], np.float32), (m, n_bins))
    assert np.array_equal(host.load(odd, 60), gpu.load_gpu(odd, 60))
    host.close()
    gpu.close()


def test_gpu_paths_match_brute_force():
    """On a five-edge diamond, every trip's GPU route is an earliest-arrival
    path among all simple paths, from the middle of its period, and its time
    is that path's from the trip's own departure."""
    from test_assign_cpu import _all_paths, _arrival, _diamond
    from paper_2406_08496_gb300.assignment import Assignment
    net, edges = _diamond()
    rng = np.random.default_rng(5)
    n_bins, bin_steps, dt, period = 6, 20, 0.5, 10
    bin_s = bin_steps * dt
    dep = np.array([0, 13, 31, 55, 70], np.uint32)
    for _ in range(20):
        tt = rng.uniform(1.0, 30.0, (6, n_bins)).astype(np.float32)
        dem = {"orig": np.zeros(5, np.uint32), "dest": np.full(5, 3, np.uint32), "depart_step": dep,
               "route_off": np.arange(0, 11, 2, dtype=np.uint64), "route_edges": np.array([0, 1] * 5, np.uint32)}
        a = Assignment(net, dem, dt=dt, seed=3)
        tsp = a.shortest_paths_gpu(tt, bin_steps, period)
        a.reroute(1.0, 0)
        routes = a.routes()
        for j in range(5):
            t0 = ((dep[j] // period) + 0.5) * period * dt
            best = min(_arrival(p, t0, tt, bin_s) for p in _all_paths(edges, 0, 3))
            r = list(routes["route_edges"][int(routes["route_off"][j]):int(routes["route_off"][j + 1])])
            assert _arrival(r, t0, tt, bin_s) == best
            tj = float(dep[j]) * dt
            assert abs(tsp[j] - (_arrival(r, tj, tt, bin_s) - tj)) < 1e-3
        a.close()


def test_msa_plain_reduces_gap(case):
    from paper_2406_08496_gb300.assignment import msa
    net, dem = case
    r = msa(net, dem, "plain", iterations=4, target_gap=0.0)
    gaps = [h["gap"] for h in r["history"]]
    assert all(g is not None and np.isfinite(g) for g in gaps)
    assert gaps[-1] < gaps[0]
    assert all(h["trips_used"] == len(dem["depart_step"]) for h in r["history"])


def test_msa_surrogate_runs_and_is_judged_by_simulation(case):
    from paper_2406_08496_gb300.assignment import msa
    net, dem = case
    r = msa(net, dem, "surrogate", iterations=5, target_gap=0.0, surrogate_batch=2048, surrogate_steps=300)
    kinds = [h["kind"] for h in r["history"]]
    assert kinds == ["simulation", "surrogate", "simulation", "surrogate", "simulation"]
    sims = [h for h in r["history"] if h["kind"] == "simulation"]
    assert all(np.isfinite(h["gap"]) for h in sims)
    assert all(np.isfinite(h["surrogate_loss"]) for h in sims)
    assert sims[-1]["gap"] < sims[0]["gap"]


def _surrogate_vs_stale(net, dem, fraction, n_pairs, batch):
    """Simulate the routes n_pairs + 1 times, `fraction` of the trips moved
    to their shortest paths between simulations; train the surrogate as the
    assignment loop does (pairs (0 -> 0), (0 -> 1), ..., (n-2 -> n-1): the
    change of each measured cell's log travel-time ratio from the earlier
    simulation, from the later routes loaded under the earlier link times and
    the earlier occupancy, ratios and inflows), predict simulation n from
    n - 1, and return the per-vehicle link-time errors (seconds; cells
    weighted by the vehicles that crossed them) of the prediction, of the
    free-flow times and of simulation n - 1's own times (the input plain MSA
    re-routes with), over every measured cell and over the cells whose
    loaded inflow changed by 10% or more."""
    from paper_2406_08496_gb300 import Simulation, Surrogate
    from paper_2406_08496_gb300.assignment import Assignment
    nb = 96
    A = Assignment(net, dem, seed=1)
    sims = []
    for k in range(n_pairs + 1):
        s = Simulation(net, dict(bin_steps=1800, n_bins=nb))
        s.load_demand(A.routes())
        s.run(300_000)
        ls = s.link_stats()
        s.close()
        tt, lr = A.link_times(ls["tt_sum"], ls["tt_cnt"])
        # these routes loaded under the earlier simulation's times (their own at first)
        loaded = A.load_gpu(sims[-1]["tt"] if sims else tt, 1800)
        sims.append(dict(ls, tt=tt, lr=lr, loaded=loaded, loaded_self=A.load_gpu(tt, 1800)))
        if k < n_pairs:
            A.shortest_paths_gpu(tt, 1800, 3600)
            A.reroute(fraction, k)
    base = [np.nan_to_num(x["lr"], nan=0.0).reshape(-1) for x in sims]
    mlp = Surrogate(n_features=11, batch=batch, seed=3)
    for ref, k in [(0, 0)] + [(k - 1, k) for k in range(1, n_pairs)]:
        r, x = sims[ref], sims[k]
        rows = np.flatnonzero(x["tt_cnt"].reshape(-1) >= 2)
        X = A.features(x["loaded_self"] if ref == k else x["loaded"], r["occ"], r["lr"], r["inflow"], rows=rows)
        mlp.pool_add(X, x["lr"].reshape(-1)[rows] - base[ref][rows])
    mlp.train_pool(1500, lr=1e-3, seed=4)
    r, x = sims[n_pairs - 1], sims[n_pairs]
    y = mlp.forward(A.features(x["loaded"], r["occ"], r["lr"], r["inflow"])) + base[n_pairs - 1]
    pred = A.times_from_ratio(y, nb).reshape(-1)
    ff = np.repeat((net["edge_len"] / net["edge_vmax"])[:, None], nb, axis=1).reshape(-1)
    w = x["tt_cnt"].reshape(-1).astype(np.float64)
    lp, lq = x["loaded"].reshape(-1).astype(np.float64), r["loaded_self"].reshape(-1).astype(np.float64)
    changed = np.abs(lp - lq) >= 0.1 * np.maximum(lq, 1.0)
    out = {}
    for name, m in (("all", w > 0), ("changed", (w > 0) & changed)):
        err = lambda p: float(np.average(np.abs(p[m] - x["tt"].reshape(-1)[m]), weights=w[m]))
        out[name] = dict(surrogate=err(pred), free_flow=err(ff), stale=err(r["tt"].reshape(-1)))
    return out


def test_surrogate_pipeline_beats_free_flow(case):
    """The loop's training and prediction path end to end on the small
    case: the prediction is far closer to the next simulation than free flow.
    (On this lightly loaded network link times hardly respond to the moved
    trips -- the change of a cell's log ratio correlates about 0.1 with the
    change of its inflow -- so the earlier simulation's own times are the
    better guess there; the regional day below is where the surrogate has
    something to predict.)"""
    e = _surrogate_vs_stale(*case, fraction=0.2, n_pairs=3, batch=2048)["all"]
    print("tiny case, link-time error per vehicle (s):", {k: round(v, 3) for k, v in e.items()})
    assert e["surrogate"] < 0.5 * e["free_flow"]


def test_surrogate_beats_stale_times_on_the_regional_day():
    """The gain of the trained network over the method without it, on the
    2.82M-trip regional day (224k nodes) with the loop's 10% re-routing:
    its prediction of the next simulation's link times is closer than the
    last simulation's own times (the input plain MSA re-routes with) over
    every measured cell, and by more on the cells whose inflow the moved
    trips changed; both far closer than free flow."""
    net, dem = W.assignment_case(scale="paper")
    import torch
    batch = 128 * 8 * torch.cuda.get_device_properties(0).multi_processor_count
    e = _surrogate_vs_stale(net, dem, fraction=0.1, n_pairs=4, batch=batch)
    print("regional day, link-time error per vehicle (s):",
          {k: {q: round(v, 3) for q, v in d.items()} for k, d in e.items()})
    assert e["all"]["surrogate"] < e["all"]["stale"] < 0.5 * e["all"]["free_flow"]
    assert e["changed"]["surrogate"] < e["changed"]["stale"]


@pytest.mark.parametrize("n_nodes", [6, 600])
def test_gpu_paths_past_the_last_millisecond(n_nodes):
    """Links shut for longer than the 32-bit milliseconds last (times past
    2^31 ms, two of them in a row on a one-way road): arrivals stop at the last
    millisecond, a trip to a node behind it still has its path, and the GPU
    search returns the host's."""
    from paper_2406_08496_gb300.assignment import Assignment
    m = n_nodes - 1
    net = {"n_nodes": n_nodes, "n_edges": m, "edge_src": np.arange(m, dtype=np.uint32),
           "edge_dst": np.arange(1, m + 1, dtype=np.uint32), "edge_len": np.full(m, 100.0, np.float32),
           "edge_lanes": np.ones(m, np.uint8), "edge_vmax": np.full(m, 10.0, np.float32)}
    dest = np.arange(1, n_nodes, dtype=np.uint32)
    n = len(dest)
    dem = {"orig": np.zeros(n, np.uint32), "dest": dest, "depart_step": np.arange(n, dtype=np.uint32),
           "route_off": np.arange(n + 1, dtype=np.uint64), "route_edges": np.zeros(n, np.uint32)}
    for n_bins in (1, 4):
        tt = np.full((m, n_bins), 20.0, np.float32)
        tt[1:3] = 3e6
        host, gpu = Assignment(net, dem, seed=1), Assignment(net, dem, seed=1)
        th, rh = _paths(host, host.shortest_paths, tt, 1800, 3600)
        tg, rg = _paths(gpu, gpu.shortest_paths_gpu, tt, 1800, 3600)
        assert np.array_equal(th.view(np.uint32), tg.view(np.uint32))
        assert np.array_equal(rh["route_off"], rg["route_off"])
        assert np.array_equal(rh["route_edges"], rg["route_edges"])
        host.close()
        gpu.close()


@pytest.mark.parametrize("side", [79, 80, 102, 103, 115, 116, 134, 135, 165, 166])
def test_gpu_paths_where_the_block_changes(side):
    """Lattices on both sides of the sizes at which the search takes another
    block (six thousand to twenty-eight thousand nodes), shuffled edge ids
    and many ties: routes and times equal the host's bit for bit."""
    _, src, dst = _lattice(side)
    _compare_paths(side * side, src, dst, 4)


@pytest.mark.parametrize("degree", [5, 8, 9])
def test_gpu_paths_with_many_out_edges(degree):
    """Up to five, eight and nine out-edges a node: rows of eight, full rows of
    eight, and none (positions through the offsets), shuffled, with ties."""
    side = 41
    _, src, dst = _lattice(side)
    i = np.arange(side * side)
    r, c = np.divmod(i, side)
    for k, (dr, dc) in enumerate([(1, 1), (-1, -1), (1, -1), (-1, 1), (2, 1)][:degree - 4]):
        m = (0 <= r + dr) & (r + dr < side) & (0 <= c + dc) & (c + dc < side)
        src, dst = np.concatenate([src, i[m]]), np.concatenate([dst, i[m] + dr * side + dc])
    assert np.bincount(src).max() == degree
    _compare_paths(side * side, src, dst, 33)


def _compare_paths(n, src, dst, n_bins):
    from paper_2406_08496_gb300.assignment import Assignment
    rng = np.random.default_rng(n)
    p = rng.permutation(len(src))
    src, dst, m = src[p].astype(np.uint32), dst[p].astype(np.uint32), len(p)
    o = rng.integers(0, n, 12).repeat(8)
    d = rng.integers(0, n, len(o))
    d = np.where(d == o, (d + 1) % n, d)
    net = {"n_nodes": n, "n_edges": m, "edge_src": src, "edge_dst": dst, "edge_len": np.full(m, 100.0, np.float32),
           "edge_lanes": np.ones(m, np.uint8), "edge_vmax": np.full(m, 10.0, np.float32)}
    dem = {"orig": o.astype(np.uint32), "dest": d.astype(np.uint32),
           "depart_step": rng.integers(0, 4000, len(o)).astype(np.uint32),
           "route_off": np.arange(len(o) + 1, dtype=np.uint64), "route_edges": np.zeros(len(o), np.uint32)}
    tt = rng.integers(1, 4, (m, n_bins)).astype(np.float32)
    host, gpu = Assignment(net, dem, seed=1), Assignment(net, dem, seed=1)
    for period in (600, 7):
        th, rh = _paths(host, host.shortest_paths, tt, 60, period)
        tg, rg = _paths(gpu, gpu.shortest_paths_gpu, tt, 60, period)
        assert np.array_equal(th.view(np.uint32), tg.view(np.uint32))
        assert np.array_equal(rh["route_off"], rg["route_off"])
        assert np.array_equal(rh["route_edges"], rg["route_edges"])
        assert np.array_equal(host.load(tt, 60), gpu.load_gpu(tt, 60))
    host.close()
    gpu.close()


def test_gpu_load_follows_every_rerouting(case):
    """Loadings on the GPU between re-routings of every size (new routes behind
    the old ones, all anew when there is no room, two re-routings between two
    loadings) count what the host walk counts."""
    from paper_2406_08496_gb300.assignment import Assignment
    net, dem = case
    A = Assignment(net, dem, seed=2)
    for it, f in enumerate([0.01, 0.02, 0.3, 0.05, 0.1, 0.1, 0.1, 1.0, 0.01, 0.6, 0.03]):
        tt = _tables(net, 96, 20 + it)
        A.shortest_paths_gpu(tt, 1800, 3600)
        A.reroute(f, it)
        if it % 4 == 1:
            continue
        assert np.array_equal(A.load(tt, 1800), A.load_gpu(tt, 1800)), it
    A.close()
