"""The calls this framework is timed on: what a user has it do, through its public entry points.

Five cases simulate (a few interactive steps, a whole demand from construction to
statistics, windows of a town's and of a regional network's rush hour, a batch of
scenarios), four run the link-travel-time surrogate (inference on a few and on many
rows, one gradient, Adam steps on the training pool) and three are the searches and
the route loading of the traffic-assignment loop.

Networks are lattices with the road classes of the repository's regional generator
(lines of local, collector, arterial and highway links; lognormal lengths; signals
where major roads meet) or its uniform signalised grid.  Trips run along major roads:
from their origin's row to an arterial column, an arterial row, another arterial
column and their destination's row, so every route is known without a search and a
large demand is drawn in milliseconds on the GPU.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2406_08496_gb300 as L
from paper_2406_08496_gb300.assignment import Assignment

DT = 0.5               # seconds per step
BIN_STEPS = 1800       # 15-minute statistics and link-time bins
N_BINS = 96            # a day of them
PERIOD_STEPS = 3600    # trips of one origin share a shortest-path tree per 30 minutes
LANES = np.array([1, 2, 3, 4], np.uint8)                    # local, collector, arterial, highway
SPEED = np.array([11.1, 15.6, 22.2, 30.0], np.float32)      # m/s
PARAM_SHAPES = dict(W1=(256, 64), b1=(256,), W2=(256, 256), b2=(256,), W3=(256, 256), b3=(256,), W4=(1, 256), b4=(1,))

# a car, a truck and a bus: acceleration, braking, standstill gap, headway, top speed
VEHICLE_TYPES = [dict(a=1.0, b=1.5, s0=2.0, T=1.5, vmax=60.0), dict(a=0.6, b=1.2, s0=3.0, T=2.0, vmax=22.0),
                 dict(a=0.8, b=1.4, s0=2.5, T=1.8, vmax=12.5)]

_allocator = []


def _start() -> None:
    # device memory from PyTorch's caching allocator, as the README and the benchmark use the library (set once:
    # contexts keep the callbacks they were made with)
    if not _allocator:
        _allocator.append(L.use_torch_allocator())


def _device() -> str:
    return "cuda" if torch.cuda.is_available() else "cpu"


# --------------------------------------------------------------------------------------
# networks and trips
# --------------------------------------------------------------------------------------

def _line_class(n: int) -> np.ndarray:
    i = np.arange(n)
    c = np.zeros(n, np.int64)
    c[i % 4 == 0] = 1
    c[i % 10 == 0] = 2
    c[i % 40 == 0] = 3
    return c


def _network(rows: int, cols: int, style: str, rng: np.random.Generator) -> tuple[dict, dict]:
    """A network and its layout: edge id of every (node, direction up / left /
    right / down), the major lines and the arterial lines.  "roads": classes by
    line, two thirds of the local links missing, two-phase signals where major
    roads meet; "grid": uniform 400 m two-lane streets, a phase per approach.
    Which links there are follows from the size alone, their lengths from rng."""
    n = rows * cols
    which = np.random.default_rng([rows, cols])
    r, c = np.divmod(np.arange(n), cols)
    grid = style == "grid"
    rc, cc = _line_class(rows), _line_class(cols)
    right, down = c < cols - 1, r < rows - 1
    h_cls, v_cls = rc[r], cc[c]
    if grid:
        h_len = v_len = np.full(n, 400.0)
        h_keep, v_keep = right, down
    else:
        h_len, v_len = np.clip(np.exp(math.log(150.0) + 0.6 * rng.standard_normal((2, n))), 10.0, 2000.0)
        h_keep = right & ((h_cls > 0) | (which.random(n) < 0.32))
        v_keep = down & ((v_cls > 0) | (which.random(n) < 0.32))

    def before(a, k):  # the value of the node k positions earlier (0 at the start)
        return np.concatenate([np.zeros(min(k, n), a.dtype), a[:n - k]])

    # out-edges of every node in ascending order of their head
    keep = np.stack([before(v_keep, cols), before(h_keep, 1), h_keep, v_keep], 1)
    length = np.stack([before(v_len, cols), before(h_len, 1), h_len, v_len], 1)
    cls = np.stack([before(v_cls, cols), before(h_cls, 1), h_cls, v_cls], 1)
    head = np.arange(n)[:, None] + np.array([-cols, -1, 1, cols])
    flat = keep.reshape(-1)
    eid = (np.cumsum(flat) - 1).reshape(n, 4)
    src = np.repeat(np.arange(n), keep.sum(1))
    dst, cls, length = head.reshape(-1)[flat], cls.reshape(-1)[flat], length.reshape(-1)[flat]
    vertical = np.tile(np.array([1, 0, 0, 1]), n)[flat]
    net = {"n_nodes": n, "n_edges": len(src), "edge_src": src.astype(np.uint32), "edge_dst": dst.astype(np.uint32),
           "edge_len": length.astype(np.float32)}
    if grid:
        net["edge_lanes"] = np.full(len(src), 2, np.uint8)
        net["edge_vmax"] = np.full(len(src), 13.9, np.float32)
        net["node_green"] = np.where(np.bincount(dst, minlength=n) >= 3, 60, 0).astype(np.uint32)
        major_r, major_c = np.arange(rows), np.arange(cols)
    else:
        net["edge_lanes"], net["edge_vmax"] = LANES[cls], SPEED[cls]
        net["node_green"] = np.where(np.bincount(dst[cls > 0], minlength=n) >= 3, 60, 0).astype(np.uint32)
        has_x = np.bincount(dst[vertical == 0], minlength=n) > 0
        net["edge_approach_rank"] = np.where(has_x[dst], vertical, 0).astype(np.uint8)
        major_r, major_c = np.flatnonzero(rc > 0), np.flatnonzero(cc > 0)
    return net, {"cols": cols, "eid": eid, "major_r": major_r, "major_c": major_c}


def _snap(lines: np.ndarray, x: np.ndarray) -> np.ndarray:
    """The major line nearest to position x."""
    i = np.clip(np.searchsorted(lines, x), 1, len(lines) - 1)
    return np.where(x - lines[i - 1] <= lines[i] - x, lines[i - 1], lines[i])


def _trips(lay: dict, n: int, rng: np.random.Generator, depart: np.ndarray, reach: float, n_access: int = 0) -> dict:
    """n trips between major intersections, `reach` lattice lines apart in each
    direction on average, from n_access origins of uneven population (0: from
    anywhere)."""
    mr, mc, cols = lay["major_r"], lay["major_c"], lay["cols"]
    if n_access:
        ar, ac = mr[rng.integers(0, len(mr), n_access)], mc[rng.integers(0, len(mc), n_access)]
        weight = np.exp(rng.standard_normal(n_access))
        pick = np.searchsorted(np.cumsum(weight) / weight.sum(), rng.random(n)).clip(0, n_access - 1)
        r0, c0 = ar[pick], ac[pick]
    else:
        r0, c0 = mr[rng.integers(0, len(mr), n)], mc[rng.integers(0, len(mc), n)]
    r1, c1 = _snap(mr, r0 + rng.laplace(0.0, reach, n)), _snap(mc, c0 + rng.laplace(0.0, reach, n))
    other = np.where(c0 == mc[-1], mc[-2], mc[np.minimum(np.searchsorted(mc, c0) + 1, len(mc) - 1)])
    c1 = np.where((r0 == r1) & (c0 == c1), other, c1)

    def toward(a, b):  # the first arterial line (every tenth) from a on the way to b, or a
        up, dn = -(-a // 10) * 10, a // 10 * 10
        return np.where((b >= a) & (up <= b), up, np.where((b < a) & (dn >= b), dn, a))

    ca, cb = toward(c0, c1), toward(c1, c0)
    both = (np.sign(cb - ca) == np.sign(c1 - c0)) & (ca != cb)
    cb = np.where(both, cb, ca)
    mid = toward(r0 + (r1 - r0) // 2, r1)
    mid = np.where(mid == r0 + (r1 - r0) // 2, r1, mid)  # no arterial row on the way: turn at the last row
    mid = np.where(both, mid, r1)
    # five legs: along the first row, a column, a row, a column, the last row
    frm = np.stack([r0 * cols + c0, r0 * cols + ca, mid * cols + ca, mid * cols + cb, r1 * cols + cb], 1)
    delta = np.stack([ca - c0, mid - r0, cb - ca, r1 - mid, c1 - cb], 1)
    dev = _device()
    d = torch.from_numpy(delta.reshape(-1)).to(dev)
    f = torch.from_numpy(frm.reshape(-1)).to(dev)
    count = d.abs()
    start = torch.cumsum(count, 0) - count
    along = torch.tensor([1, cols, 1, cols, 1], device=dev).repeat(n)
    step = torch.sign(d) * along
    # direction index: up 0, left 1, right 2, down 3
    turn = torch.where(along == 1, torch.where(d < 0, 1, 2), torch.where(d < 0, 0, 3))
    if cols == 1:
        raise ValueError("a lattice has at least two columns")
    leg = torch.repeat_interleave(torch.arange(5 * n, device=dev), count)
    at = torch.arange(leg.numel(), device=dev) - start[leg]
    eid = torch.from_numpy(lay["eid"]).to(dev)
    edges = eid.reshape(-1)[(f[leg] + at * step[leg]) * 4 + turn[leg]].to(torch.int32).cpu().numpy().view(np.uint32)
    off = np.zeros(n + 1, np.uint64)
    off[1:] = torch.cumsum(count.reshape(n, 5).sum(1), 0).cpu().numpy()
    return {"orig": (r0 * cols + c0).astype(np.uint32), "dest": (r1 * cols + c1).astype(np.uint32),
            "depart_step": depart.astype(np.uint32), "route_off": off, "route_edges": edges}


def _day_departures(n: int, rng: np.random.Generator) -> np.ndarray:
    """A day's departure steps: half around 08:00, half around 17:30."""
    t = np.where(rng.random(n) < 0.5, 8.0, 17.5) + 0.75 * rng.standard_normal(n)
    return np.ceil(np.clip(t, 0.0, 23.9) * 3600.0 / DT)


REACH = 25.0  # lattice lines a trip wants to cover in each direction, on average (the network's edge cuts some short)
LINK_STEPS = {"roads": 24.0, "grid": 110.0}  # steps per link at a window's load, signals included, about
WARM_STEPS = 3072  # steps before a window: the network has filled


def _links(rows: int, cols: int, reach: float) -> float:
    """Links of a trip on a lattice, about."""
    return reach * (rows / (rows + 2.0 * reach) + cols / (cols + 2.0 * reach))


def _window_demand(lay: dict, style: str, vehicles: int, rng: np.random.Generator, horizon: int) -> dict:
    """Steady departures that keep about `vehicles` on the network."""
    rows, cols = len(lay["eid"]) // lay["cols"], lay["cols"]
    n = max(8, int(vehicles * horizon / (LINK_STEPS[style] * _links(rows, cols, REACH))))
    return _trips(lay, n, rng, rng.integers(0, horizon, n), REACH)


# --------------------------------------------------------------------------------------
# surrogate inputs and the same network in 64 bits
# --------------------------------------------------------------------------------------

def _weights(features: int, rng: np.random.Generator) -> dict:
    """Parameters of a model in use: scaled normal weights, small biases."""
    p = {}
    for k, s in PARAM_SHAPES.items():
        fan = features if k == "W1" else 256
        p[k] = (rng.standard_normal(s) * (math.sqrt(2.0 / fan) if k[0] == "W" else 0.1)).astype(np.float32)
    p["W1"][:, features:] = 0.0
    return p


def _samples(rows: int, features: int, seed: int) -> tuple[np.ndarray, np.ndarray]:
    """Inputs scaled as the surrogate's features are (lengths, log inflows and
    densities of order one) and the log travel-time ratio changes to learn."""
    dev = _device()
    gen = torch.Generator(dev).manual_seed(seed)
    X = torch.randn((rows, features), device=dev, generator=gen).mul_(0.7).add_(0.3)
    t = 0.3 * torch.sin(2.0 * X[:, 0]) + 0.2 * X[:, features // 2] + \
        0.1 * torch.randn(rows, device=dev, generator=gen)
    return X.cpu().numpy(), t.cpu().numpy()


def _forward64(p: dict, X: torch.Tensor) -> torch.Tensor:
    h = X
    for w, b in (("W1", "b1"), ("W2", "b2"), ("W3", "b3")):
        W = p[w][:, :X.shape[1]] if w == "W1" else p[w]
        h = torch.nn.functional.gelu(h @ W.T + p[b])
    return (h @ p["W4"].T).reshape(-1) + p["b4"]


def _params64(p: dict) -> dict:
    return {k: torch.from_numpy(v).to(_device(), torch.float64) for k, v in p.items()}


def _loss_grads64(p: dict, X: torch.Tensor, t: torch.Tensor) -> tuple[torch.Tensor, dict]:
    q = {k: v.detach().requires_grad_(True) for k, v in p.items()}
    loss = torch.mean((_forward64(q, X) - t) ** 2)
    loss.backward()
    return loss.detach(), {k: v.grad for k, v in q.items()}


def _mix64(z: np.ndarray) -> np.ndarray:
    z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
    z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
    return z ^ (z >> np.uint64(31))


def _pool_rows(n: int, batch: int, step: int, seed: int) -> np.ndarray:
    """Pool rows of a training step's minibatch: the documented shuffled passes
    (a four-round Feistel network with cycle walking)."""
    h = 1
    while (1 << (2 * h)) < n:
        h += 1
    pos = np.uint64(step) * np.uint64(batch) + np.arange(batch, dtype=np.uint64)
    with np.errstate(over="ignore"):
        key = _mix64(np.uint64(seed) ^ (pos // np.uint64(n) * np.uint64(0xD1B54A32D192ED03)))
        mask, r = np.uint64((1 << h) - 1), pos % np.uint64(n)
        todo = np.ones(batch, bool)
        while todo.any():
            hi, lo, k = r[todo] >> np.uint64(h), r[todo] & mask, key[todo]
            for i in range(4):
                f = _mix64(k ^ np.uint64((0x9E3779B97F4A7C15 * (i + 1)) % (1 << 64)) ^ lo) & mask
                hi, lo = lo, hi ^ f
            r[todo] = (hi << np.uint64(h)) | lo
            todo = r >= np.uint64(n)
    return r.astype(np.int64)


# --------------------------------------------------------------------------------------
# cases
# --------------------------------------------------------------------------------------

def listed() -> list[dict]:
    return [
        # a user stepping a small signalised grid and looking at it, with trucks and buses, overtaking and noisy gaps
        dict(name="steps_grid", kind="steps", style="grid", rows=8, cols=8, trips=300, steps=37),
        # a whole demand on the 8x8 grid, from construction to the trip table and link statistics
        dict(name="run_grid", kind="run", style="grid", rows=8, cols=8, trips=2000, over=3600),
        # the rush hour of a town (27k-node lattice): 17 minutes, not a whole number of chunks
        dict(name="window_town", kind="window", rows=165, cols=165, vehicles=13000, steps=2000),
        # the rush hour of a region (224k nodes): 12.8 minutes of a quarter of a million vehicles
        dict(name="window_region", kind="window", rows=473, cols=474, vehicles=250000, steps=1536),
        # independent scenarios of uneven size advanced together
        dict(name="window_batch", kind="batch", scenarios=24, rows=30, cols=70, vehicles=60000, steps=1536),
        # scoring a few hundred links with the surrogate
        dict(name="forward_997", kind="forward", rows=997, features=11, batch=8192),
        # scoring every (link, bin) cell of part of a network, at the loop's default batch
        dict(name="forward_2m", kind="forward", rows=2000003, features=11, batch=8192),
        # the gradient of one batch (a caller that averages gradients itself)
        dict(name="grad_8k", kind="grad", rows=8000, features=11, batch=8192),
        # twenty Adam steps on the training pool
        dict(name="train_8k", kind="train", pool=200003, features=11, batch=8192, steps=20),
        # all-or-nothing assignment of a small network's trips: search, move every trip, propagate the new routes
        dict(name="reroute_small", kind="reroute", rows=50, cols=55, trips=30000, access=60),
        # time-dependent shortest paths of a town's day
        dict(name="paths_town", kind="paths", rows=165, cols=165, trips=340000, access=384),
        # a town's routes propagated with given link times
        dict(name="load_town", kind="load", rows=165, cols=165, trips=340000, access=384),
    ]


def draw(rng) -> dict:
    def log(lo: float, hi: float) -> int:
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["steps", "run", "window", "batch", "forward", "forward", "grad", "train", "reroute", "paths",
                       "load"])
    if kind == "steps":
        return dict(kind=kind, style=rng.choice(["grid", "roads"]), rows=rng.randint(9, 24), cols=rng.randint(9, 24),
                    trips=log(20, 1200), steps=log(1, 200))
    if kind == "run":
        side = rng.randint(6, 24)
        return dict(kind=kind, style="grid", rows=side, cols=rng.randint(6, 24), trips=log(300, 6000),
                    over=log(900, 5400))
    if kind == "window":
        rows, cols = log(60, 470), log(60, 470)
        return dict(kind=kind, rows=rows, cols=cols, vehicles=max(500, int(rows * cols * rng.uniform(0.2, 1.1))),
                    steps=log(100, 1536))
    if kind == "batch":
        n = log(2, 40)
        return dict(kind=kind, scenarios=n, rows=rng.randint(20, 40), cols=rng.randint(40, 80),
                    vehicles=n * log(500, 3000), steps=log(200, 1536))
    if kind == "forward":
        return dict(kind=kind, rows=log(1, 2000000), features=rng.choice([9, 11, 11, rng.randint(1, 64)]),
                    batch=128 * log(1, 1216))
    if kind == "grad":
        batch = 128 * log(1, 256)
        return dict(kind=kind, rows=rng.randint(max(1, batch // 2), batch), features=rng.choice([9, 11, 33]),
                    batch=batch)
    if kind == "train":
        return dict(kind=kind, pool=log(500, 400000), features=rng.choice([9, 11]), batch=128 * log(8, 160),
                    steps=rng.randint(1, 20))
    rows, cols = log(24, 165), log(24, 165)
    trips = max(200, int(rows * cols * rng.uniform(3.0, 12.0)))
    return dict(kind=kind, rows=rows, cols=cols, trips=trips, access=max(8, rows * cols // 70))


def work(case: dict) -> dict:
    k = case["kind"]
    if k in ("forward", "grad", "train"):
        mac = case["features"] * 256 + 2 * 256 * 256 + 256
        rows = case["rows"] if k != "train" else min(case["pool"], case["batch"]) * case["steps"]
        n_par = 4 * sum(math.prod(s) for s in PARAM_SHAPES.values())
        inp = rows * 4 * (case["features"] + 1)
        return {"bytes": inp + n_par * {"forward": 1, "grad": 2, "train": 6 * case.get("steps", 1)}[k],
                "flops": 2.0 * mac * rows * (1 if k == "forward" else 3)}
    if k in ("steps", "run", "window", "batch"):
        # a vehicle's step reads and writes its state and reads the cells ahead of it: 64 bytes
        if k == "steps":
            veh_steps = 0.6 * case["trips"] * case["steps"]
        elif k == "run":
            # 400 m links: half a minute each and half a minute at its signal
            veh_steps = 120.0 * case["trips"] * _links(case["rows"], case["cols"], min(6.0, case["rows"] / 3.0))
        else:
            veh_steps = float(case["vehicles"]) * case["steps"]
        return {"bytes": 64.0 * veh_steps, "flops": 40.0 * veh_steps}
    # link-time tables in, one path (or one walk) per trip: edge ids and link times
    edges = 2.1 * case["rows"] * case["cols"]
    steps = case["trips"] * _links(case["rows"], case["cols"], min(REACH, (case["rows"] + case["cols"]) / 6.0))
    return {"bytes": edges * N_BINS * 4.0 * (2 if k == "load" else 1) + 12.0 * steps, "flops": 2.0 * steps}


def prepare(case: dict, seed: int):
    _start()
    k = case["kind"]
    rng = np.random.default_rng([seed, 2406])
    if k in ("forward", "grad", "train"):
        m = L.Surrogate(n_features=case["features"], batch=case["batch"], seed=seed)
        p = _weights(case["features"], rng)
        m.set_params(p)
        rows = case["pool"] if k == "train" else case["rows"]
        X, t = _samples(rows, case["features"], seed)
        if k == "train":
            m.pool_add(X, t)
        return dict(kind=k, model=m, params=p, X=X, t=t, seed=seed, steps=case.get("steps", 0))
    if k == "steps":
        net, lay = _network(case["rows"], case["cols"], case["style"], rng)
        n = case["trips"]
        dem = _trips(lay, n, rng, rng.integers(0, 40, n), 3.0)
        dem["vtype"] = rng.choice(3, n, p=[0.85, 0.1, 0.05]).astype(np.uint8)
        sim = L.Simulation(net, dict(bin_steps=BIN_STEPS, n_bins=4, seed=seed, eps_amp=1.0, dlc_prob=0.3, dlc_gain=3.0),
                           vehicle_types=VEHICLE_TYPES)
        sim.load_demand(dem)
        return dict(kind=k, sim=sim, steps=case["steps"])
    if k == "run":
        net, lay = _network(case["rows"], case["cols"], case["style"], rng)
        dem = _trips(lay, case["trips"], rng, rng.integers(0, case["over"], case["trips"]), min(6.0, case["rows"] / 3.0))
        return dict(kind=k, net=net, dem=dem, seed=seed)
    if k == "window":
        net, lay = _network(case["rows"], case["cols"], "roads", rng)
        sim = L.Simulation(net, dict(bin_steps=BIN_STEPS, n_bins=4, seed=seed))
        sim.load_demand(_window_demand(lay, "roads", case["vehicles"], rng, WARM_STEPS + case["steps"]))
    elif k == "batch":
        nets, dems = [], []
        size = np.exp(np.random.default_rng(case["scenarios"]).uniform(-1.0, 1.0, case["scenarios"]))
        for s in range(case["scenarios"]):
            f = math.sqrt(size[s])
            style = "roads" if s % 2 else "grid"
            net, lay = _network(max(9, int(case["rows"] * f)), max(9, int(case["cols"] * f)), style, rng)
            nets.append(net)
            dems.append(_window_demand(lay, style, int(case["vehicles"] * size[s] / size.sum()), rng,
                                       WARM_STEPS + case["steps"]))
        sim = L.BatchSimulation(nets, dict(bin_steps=BIN_STEPS, n_bins=4))
        sim.load_demand(dems, seeds=rng.integers(1, 1 << 40, case["scenarios"]))
    else:
        net, lay = _network(case["rows"], case["cols"], "roads", rng)
        n = case["trips"]
        dem = _trips(lay, n, rng, _day_departures(n, rng), min(REACH, (case["rows"] + case["cols"]) / 6.0),
                     case["access"])
        # link times of a day: the free-flow time, longer by up to a factor of 3 around the peaks
        dev = _device()
        gen = torch.Generator(dev).manual_seed(seed)
        hour = (torch.arange(N_BINS, device=dev) + 0.5) * BIN_STEPS * DT / 3600.0
        peak = torch.exp(-0.5 * ((hour - 8.0) / 1.0) ** 2) + torch.exp(-0.5 * ((hour - 17.5) / 1.2) ** 2)
        busy = torch.rand((net["n_edges"], 1), device=dev, generator=gen) * peak
        noise = torch.rand((net["n_edges"], N_BINS), device=dev, generator=gen)
        ff = torch.from_numpy(net["edge_len"] / net["edge_vmax"]).to(dev)
        tt = (ff[:, None] * (1.0 + 2.0 * busy + 0.2 * noise)).cpu().numpy()
        return dict(kind=k, engine=Assignment(net, dem, dt=DT, seed=seed), tt=tt)
    sim.step(WARM_STEPS)
    sim.snapshot()
    return dict(kind=k, sim=sim, steps=case["steps"])


def run(state):
    k = state["kind"]
    if k == "forward":
        return state["model"].forward(state["X"])
    if k == "grad":
        loss, grads = state["model"].grad(state["X"], state["t"])
        return {"loss": loss, "grads": grads}
    if k == "train":
        m = state["model"]
        m.set_params(state["params"])
        losses = m.train_pool(state["steps"], lr=1e-3, seed=state["seed"])
        return {"losses": losses, "params": m.get_params()}
    if k == "steps":
        sim = state["sim"]
        sim.reset()
        sim.step(state["steps"])
        return sim.state()
    if k in ("window", "batch"):
        sim = state["sim"]
        sim.restore()
        sim.step(state["steps"])
        return {"state": sim.state(), "veh_steps": sim.counters()["veh_steps"]}
    if k == "run":
        sim = L.Simulation(state["net"], dict(bin_steps=BIN_STEPS, n_bins=12, seed=state["seed"]))
        vid = sim.load_demand(state["dem"])
        done = sim.run(100000)
        out = {"vid": vid, "steps": done["steps"], "veh_steps": done["veh_steps"], "trips": sim.trips(),
               "links": sim.link_stats()}
        sim.close()
        return out
    a = state["engine"]
    if k == "load":
        return a.load_gpu(state["tt"], BIN_STEPS).view(np.int32)
    tsp = a.shortest_paths_gpu(state["tt"], BIN_STEPS, PERIOD_STEPS)
    if k == "paths":
        return tsp
    moved = a.reroute(1.0, 0)
    return {"tsp": tsp, "moved": moved, "inflow": a.load_gpu(state["tt"], BIN_STEPS).view(np.int32)}


def exact(case: dict, seed: int):
    """The surrogate's outputs in 64 bits.  A simulation has no such value (its
    rules are 32-bit roundings that decide who goes first) and a search's times
    are exact sums of whole milliseconds."""
    k = case["kind"]
    if k not in ("forward", "grad", "train"):
        return None
    rng = np.random.default_rng([seed, 2406])
    p = _params64(_weights(case["features"], rng))
    dev = _device()
    X, t = _samples(case["pool"] if k == "train" else case["rows"], case["features"], seed)
    if k == "forward":
        parts = [_forward64(p, torch.from_numpy(X[i:i + 65536]).to(dev, torch.float64)) for i in
                 range(0, len(X), 65536)]
        return torch.cat(parts).cpu().numpy()
    X, t = torch.from_numpy(X).to(dev, torch.float64), torch.from_numpy(t).to(dev, torch.float64)
    if k == "grad":
        loss, g = _loss_grads64(p, X, t)
        return {"loss": float(loss), "grads": {n: v.cpu().numpy() for n, v in g.items()}}
    # Adam as lpsim_mlp_train_pool documents it
    batch = min(case["batch"], case["pool"])
    mo = {n: torch.zeros_like(v) for n, v in p.items()}
    ve = {n: torch.zeros_like(v) for n, v in p.items()}
    losses = []
    for s in range(case["steps"]):
        rows = torch.from_numpy(_pool_rows(case["pool"], batch, s, seed)).to(dev)
        loss, g = _loss_grads64(p, X[rows], t[rows])
        losses.append(float(loss))
        for n in p:
            mo[n] = 0.9 * mo[n] + 0.1 * g[n]
            ve[n] = 0.999 * ve[n] + 0.001 * g[n] ** 2
            p[n] = p[n].detach() - 1e-3 * (mo[n] / (1 - 0.9 ** (s + 1))) / \
                (torch.sqrt(ve[n] / (1 - 0.999 ** (s + 1))) + 1e-8)
    return {"losses": np.array(losses), "params": {n: v.cpu().numpy() for n, v in p.items()}}
