"""What a user of the library has it do, as measurable cases: stepping networks of every
size (graph and persistent execution, batched, with outputs and vehicle types), trip
planning, the route equilibrium, the static assignment and the calibration gradient.

Most stepping cases advance a state that keeps going from pass to pass, as a program that
watches a running simulation does (their demand keeps the number of vehicles on the road
about the same over the thousands of steps of a measurement); the queues, the outputs, the
equilibrium and the calibration start each pass from a snapshot or from empty roads, as a
forecast or an evaluation loop does."""
import functools
import math

import numpy as np
import torch

from paper_1807_01148_gb300 import gbtraffic as G
from paper_1807_01148_gb300 import scenarios as S

FIELDS = (("status", torch.uint8), ("link", torch.int32), ("lane", torch.int32), ("cursor", torch.int32),
          ("x", torch.float32), ("v", torch.float32), ("insert_step", torch.int32),
          ("arrive_step", torch.int32), ("lane_change", torch.int8))
SCHEDULE = (65536, 65536, 32768, 16384)       # the paper's decaying reroute, 1/65536 of the trips
CARS_AND_TRUCKS = ((4.5, 1.0, 40.0), (12.0, 0.6, 22.0), (18.0, 0.5, 18.0))


def listed():
    return [
        # one vehicle class on a closed single-lane road, watched every few steps: the smallest call
        dict(name="ring", kind="ring", vehicles=50, steps=10),
        # the signalised 20 x 20 grid in mid-run: a small study area, bound by launches
        dict(name="grid20", kind="grid", side=20, hourly=20000, hours=10, warm=2400, steps=20),
        # 64 uneven grid scenarios with their own drivers in one batched handle
        dict(name="ensemble64", kind="ensemble", scenarios=64, hours=2.5, warm=1500, steps=10),
        # a metropolitan network at its natural morning peak: few vehicles, many lanes, departures
        dict(name="metro_peak", kind="metro", nx=500, ny=450, trips=1400000, active=165000, hops=56, window=15000,
             loop=False, persistent=True, steps=10),
        # the same network with every trip on the road: the throughput case
        dict(name="metro_full", kind="metro", nx=500, ny=450, trips=2110000, active=2110000, hops=24, window=1,
             loop=True, persistent=False, steps=4),
        # standing queues of 285 vehicles per lane in front of signals: the next minute from the present state
        dict(name="jam1000", kind="jam", corridors=1000, lanes=2, length=2000.0, spacing=7.0, steps=120),
        # fuel, CO, traversal times and edge samples of a mixed fleet over a minute, from a snapshot
        dict(name="outputs_fleet", kind="outputs", nx=120, ny=100, trips=120000, active=90000, hops=24, steps=120),
        # trip planning on the metropolitan network, one tree per origin
        dict(name="route_metro", kind="route", nx=500, ny=450, trips=12000),
        # the four-iteration route equilibrium on a town
        dict(name="equilibrium", kind="equilibrium", nx=48, ny=40, trips=16000, steps=300),
        # the static user equilibrium of a district by Frank-Wolfe
        dict(name="assign", kind="assign", nx=120, ny=100, trips=60000, iters=3),
        # calibration: loss and gradient of the 20 x 20 grid with three link classes
        dict(name="calib_grad", kind="calib", side=20, trips=20000, steps=1800, every=20, grad=True),
        # calibration: the loss alone, as a line search asks for it
        dict(name="calib_loss", kind="calib", side=20, trips=20000, steps=600, every=20, grad=False),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["ring", "grid", "ensemble", "metro", "metro", "jam", "outputs", "route", "equilibrium",
                       "assign", "calib"])
    if kind == "ring":
        return dict(kind=kind, vehicles=_log_int(rng, 3, 400), steps=_log_int(rng, 1, 40))
    if kind == "grid":
        side = rng.randint(5, 40)
        return dict(kind=kind, side=side, hourly=50 * side * side + rng.randint(0, 999), hours=rng.randint(4, 8),
                    warm=rng.randint(600, 2400), steps=rng.randint(3, 20))
    if kind == "ensemble":
        return dict(kind=kind, scenarios=_log_int(rng, 3, 63), hours=rng.uniform(1.5, 2.5),
                    warm=rng.randint(300, 1500), steps=rng.randint(3, 10))
    if kind == "metro":
        nx, ny = _log_int(rng, 40, 500), _log_int(rng, 40, 440)
        room = 9.5 * nx * ny                  # vehicles of a full road network of this size
        active = min(2000000, _log_int(rng, max(200, room / 20), room))
        return dict(kind=kind, nx=nx, ny=ny, trips=active + rng.randint(0, 100000), active=active,
                    hops=rng.randint(12, 24), window=rng.randint(500, 6000), loop=rng.random() < 0.5,
                    persistent=rng.random() < 0.5, steps=rng.randint(2, 9))
    if kind == "jam":
        return dict(kind=kind, corridors=_log_int(rng, 10, 999), lanes=rng.randint(1, 4),
                    length=float(rng.randint(300, 2000)), spacing=rng.uniform(6.5, 12.0), steps=rng.randint(10, 120))
    if kind == "outputs":
        nx, ny = _log_int(rng, 24, 120), _log_int(rng, 20, 100)
        active = _log_int(rng, max(100, nx * ny / 2), 7 * nx * ny)
        return dict(kind=kind, nx=nx, ny=ny, trips=active + active // 3, active=active, hops=rng.randint(10, 24),
                    steps=20 * rng.randint(1, 6))
    if kind == "route":
        nx, ny = _log_int(rng, 20, 500), _log_int(rng, 20, 450)
        return dict(kind=kind, nx=nx, ny=ny, trips=_log_int(rng, 300, 11999))
    if kind == "equilibrium":
        return dict(kind=kind, nx=rng.randint(12, 48), ny=rng.randint(12, 40), trips=_log_int(rng, 500, 15999),
                    steps=rng.randint(60, 300))
    if kind == "assign":
        return dict(kind=kind, nx=_log_int(rng, 16, 120), ny=_log_int(rng, 14, 100), trips=_log_int(rng, 1000, 59999),
                    iters=rng.randint(0, 3))
    every = rng.randint(5, 25)
    return dict(kind=kind, side=rng.randint(6, 20), trips=_log_int(rng, 500, 19999), steps=every * rng.randint(4, 70),
                every=every, grad=rng.random() < 0.5)


# ---------------------------------------------------------------------------- inputs
_DEV = "cuda" if torch.cuda.is_available() else "cpu"


def _rng(seed):
    g = torch.Generator(device=_DEV)
    g.manual_seed(int(seed) * 2654435761 % (1 << 62))
    return g


@functools.lru_cache(maxsize=8)
def _metro(nx, ny):
    """The road network of a metropolitan area of nx x ny junctions (the same roads for every seed: a
    user has one map and many demands)."""
    und = int(round(275_000 * (nx * ny) / 225_000))
    return S.metro(nx=nx, ny=ny, n_undirected=max(und, nx * ny - 1), n_trips=1)


def _demand(net, first, last, depart):
    return dict(n_trips=len(first), origin=net["link_from"][first], dest=net["link_to"][last],
                depart_step=np.ascontiguousarray(depart, np.int32))


def _busy(nx, ny, trips, active, hops, window, loop, seed):
    """A metropolitan network with about `active` vehicles on the road, at most one per 8 m of lane and
    evenly spread over each lane, and the other trips departing over the next `window` steps; every trip
    follows a walk of hops/2 .. 3 hops/2 links that prefers the main roads and turns back only at dead
    ends, or with loop drives it there and back for ever (a fleet in circulation)."""
    sc = _metro(nx, ny)
    net = sc["network"]
    g = _rng(seed)
    t = lambda a, dt: torch.from_numpy(np.ascontiguousarray(a)).to(_DEV, dt)  # noqa: E731
    lf, lt = t(net["link_from"], torch.int64), t(net["link_to"], torch.int64)
    length, lanes = t(net["link_length_m"], torch.float64), t(net["link_lanes"], torch.int64)
    cls = t(net["link_class"], torch.int64)
    nl, nn = len(lf), net["n_nodes"]
    order = torch.argsort(lf, stable=True)
    deg = torch.bincount(lf, minlength=nn)
    start = torch.cumsum(deg, 0) - deg
    # vehicles of every lane
    lane_link = torch.repeat_interleave(torch.arange(nl, device=_DEV), lanes)
    lane_base = torch.cumsum(lanes, 0) - lanes
    lane_of = torch.arange(len(lane_link), device=_DEV) - lane_base[lane_link]
    cap = torch.floor(length / 8.0)[lane_link]
    share = length * torch.tensor([1.0, 3.0, 4.0], device=_DEV, dtype=torch.float64)[cls]   # traffic by road class
    mean = share[lane_link] * (active / float((share * lanes).sum()))
    count = torch.minimum(torch.poisson(mean, generator=g), cap).long()
    first_of = torch.cumsum(count, 0) - count
    lane_id = torch.repeat_interleave(torch.arange(len(count), device=_DEV), count)
    k = torch.arange(len(lane_id), device=_DEV) - first_of[lane_id]
    x = (k + 0.5) * length[lane_link[lane_id]] / count[lane_id]
    n = min(len(lane_id), active, trips)
    pick = torch.randperm(len(lane_id), generator=g, device=_DEV)[:n]
    vid = torch.randperm(trips, generator=g, device=_DEV)
    link = torch.randint(0, nl, (trips,), generator=g, device=_DEV)
    link[vid[:n]] = lane_link[lane_id[pick]]
    # the walks
    key = lf * nn + lt
    by_key = torch.argsort(key)
    twin = by_key[torch.searchsorted(key[by_key], lt * nn + lf)]      # every road has both directions
    n_hops = torch.randint(max(1, hops // 2), 3 * hops // 2 + 1, (trips,), generator=g, device=_DEV)
    legs = 2 * n_hops if loop else n_hops
    off = torch.zeros(trips + 1, dtype=torch.int64, device=_DEV)
    off[1:] = torch.cumsum(legs, 0)
    routes = torch.empty(int(off[-1]), dtype=torch.int32, device=_DEV)
    e = link.clone()
    for h in range(int(n_hops.max())):
        on = h < n_hops
        routes[(off[:-1] + h)[on]] = e[on].int()
        if loop:
            routes[(off[1:] - 1 - h)[on]] = twin[e[on]].int()
        d = deg[lt[e]]
        cand = []
        for _ in range(2):
            r = torch.randint(0, 1 << 20, (trips,), generator=g, device=_DEV) % d
            nxt = order[start[lt[e]] + r]
            back = (lt[nxt] == lf[e]) & (d > 1)
            cand.append(torch.where(back, order[start[lt[e]] + (r + 1) % d], nxt))
        e = torch.where(cls[cand[1]] > cls[cand[0]], cand[1], cand[0])
    host = lambda a, dt: a.cpu().numpy().astype(dt, copy=False)  # noqa: E731
    st = dict(status=torch.zeros(trips, dtype=torch.uint8, device=_DEV), link=torch.zeros_like(link),
              lane=torch.zeros_like(link), cursor=torch.zeros_like(link),
              x=torch.zeros(trips, device=_DEV), v=torch.zeros(trips, device=_DEV))
    on = vid[:n]
    st["status"][on] = 1
    st["link"][on] = link[on]
    st["lane"][on] = lane_of[lane_id[pick]]
    st["x"][on] = x[pick].float()
    st["v"][on] = 0.5 * t(net["link_speed_mps"], torch.float32)[link[on]]
    state = {a: host(b, np.float32 if a in "xv" else np.uint8 if a == "status" else np.int32) for a, b in st.items()}
    depart = host(torch.randint(0, window, (trips,), generator=g, device=_DEV), np.int32)
    off, routes = host(off, np.int32), host(routes, np.int32)
    dem = _demand(net, routes[off[:-1]], routes[off[1:] - 1], depart)
    return dict(sc, demand=dem, params=dict(sc["params"], loop_routes=int(loop)), routes=dict(offsets=off, links=routes), init_state=state)


def _trips(nx, ny, trips, seed, window=None):
    """The gravity demand of a metropolitan network; with window: all departing over that many steps."""
    sc = _metro(nx, ny)
    rng = np.random.default_rng([int(seed), 77])
    rad = 100.0 * np.exp(rng.uniform(-0.5, math.log(math.hypot(nx, ny) * 1.5), trips))
    th = rng.uniform(0, 2 * np.pi, trips)
    o = rng.integers(0, nx * ny, trips)
    c = np.clip(o % nx + np.rint(rad * np.cos(th) / 150.0).astype(np.int64), 0, nx - 1)
    r = np.clip(o // nx + np.rint(rad * np.sin(th) / 150.0).astype(np.int64), 0, ny - 1)
    d = r * nx + c
    d = np.where(d == o, (o + 1) % (nx * ny), d)
    dep = rng.integers(0, window or 172_800, trips)
    return dict(sc, demand=dict(n_trips=trips, origin=o.astype(np.int32), dest=d.astype(np.int32),
                                depart_step=dep.astype(np.int32)))


def _costs(net, seed):
    """Link costs (deciseconds) of a congested hour: free flow times 1 to 1.5."""
    rng = np.random.default_rng([int(seed), 78])
    ff = 10.0 * net["link_length_m"].astype(np.float64) / net["link_speed_mps"]
    return np.maximum(1, np.rint(ff * rng.uniform(1.0, 1.5, len(ff)))).astype(np.int32)


# ---------------------------------------------------------------------------- the calls
def _sim(sc, scenarios=None):
    sim = G.Sim.batch(scenarios) if scenarios else G.Sim(sc)
    if torch.cuda.is_available():
        sim.set_stream(torch.cuda.current_stream().cuda_stream)
    return sim


def _buffers(sim):
    return {k: torch.empty(sim.n_trips, dtype=dt, device=_DEV) for k, dt in FIELDS}


def prepare(case, seed):
    c = dict(case)
    kind = c["kind"]
    if kind == "ring":
        sc = S.ring(n_veh=c["vehicles"], circumference=20.0 * c["vehicles"], seed=S.BASE_SEED + seed)
        sim = G.setup(sc, _sim(sc))
        return dict(c, sim=sim, out=_buffers(sim))
    if kind == "grid":
        sim = _sim(S.grid(n=c["side"], n_trips=c["hourly"] * c["hours"], depart_window_s=3600.0 * c["hours"],
                          seed=S.BASE_SEED + seed))
        sim.route()
        sim.step(c["warm"])
        return dict(c, sim=sim, out=_buffers(sim))
    if kind == "ensemble":
        scs = S.ensemble(n_scen=c["scenarios"])       # these networks and drivers; demand by seed, at their rate
        rng = np.random.default_rng([int(seed), 80])
        for sc in scs:
            nn, n = sc["network"]["n_nodes"], int(sc["demand"]["n_trips"] * c["hours"])
            o = rng.integers(0, nn, n)
            sc["demand"] = dict(n_trips=n, origin=o, dest=(o + rng.integers(1, nn, n)) % nn,
                                depart_step=rng.integers(0, int(7200 * c["hours"]), n))
        sim = _sim(None, scs)
        sim.route()
        sim.step(c["warm"])
        return dict(c, sim=sim, out=_buffers(sim))
    if kind == "metro":
        sc = _busy(c["nx"], c["ny"], c["trips"], c["active"], c["hops"], c["window"], c["loop"], seed)
        sim = G.setup(sc, _sim(sc))
        if c["persistent"]:
            sim.set_exec(mode=G.SIM_EXEC_PERSISTENT, threads=256, blocks_per_sm=4)
        return dict(c, sim=sim, out=_buffers(sim))
    if kind == "jam":
        sc = S.jammed_corridors(n_corr=c["corridors"], lanes=c["lanes"], length=c["length"], spacing=c["spacing"],
                                seed=S.BASE_SEED + seed)
        sim = G.setup(sc, _sim(sc))
        return dict(c, sim=sim, out=_buffers(sim), start=sc["init_state"])
    if kind == "outputs":
        sc = _busy(c["nx"], c["ny"], c["trips"], c["active"], c["hops"], c["steps"], False, seed)
        sim = G.setup(sc, _sim(sc))
        rng = np.random.default_rng([int(seed), 79])
        sim.set_vehicle_types(list(CARS_AND_TRUCKS),
                              rng.choice(3, sim.n_trips, p=(0.85, 0.1, 0.05)).astype(np.uint8))
        sim.set_outputs(G.OUT_EMISSIONS | G.OUT_LINK_TIMES | G.OUT_EDGE_SAMPLES, sample_every=20, per_window=3,
                        max_windows=2)
        return dict(c, sim=sim, out=_buffers(sim), start=sc["init_state"])
    if kind == "route":
        sc = _trips(c["nx"], c["ny"], c["trips"], seed)
        room = np.zeros(c["trips"] * (c["nx"] + c["ny"]) // 2, np.int32)    # where the program keeps the paths
        return dict(c, sim=_sim(sc), costs=_costs(sc["network"], seed), paths=room)
    if kind == "equilibrium":
        sim = _sim(_trips(c["nx"], c["ny"], c["trips"], seed, window=max(1, c["steps"] // 2)))
        sim.set_outputs(G.OUT_LINK_TIMES)
        return dict(c, sim=sim, out=_buffers(sim))
    if kind == "assign":
        sc = _trips(c["nx"], c["ny"], c["trips"], seed)
        period = 24.0 * c["trips"] / 3_000_000 * 225_000 / (c["nx"] * c["ny"])   # about the metro's daily load
        return dict(c, sim=_sim(sc), capacity=S.bpr_capacity(sc, period / 8, S.METRO_EDGE_TYPES))
    sc = S.calib(steps=c["steps"], n=c["side"], n_trips=c["trips"], seed=S.BASE_SEED + seed)
    sim = _sim(sc)
    sim.route()
    n = sim.n_trips
    start = dict(status=np.zeros(n, np.uint8), link=np.zeros(n, np.int32), lane=np.zeros(n, np.int32),
                 cursor=np.zeros(n, np.int32), x=np.zeros(n, np.float32), v=np.zeros(n, np.float32))
    nominal, wanted = ([np.array(sc[p][k], np.float64) for k in G.PARAM_ORDER] for p in ("params", "target_params"))
    sim.set_class_params(*wanted)
    target = sim.observe(c["steps"], c["every"])
    return dict(c, sim=sim, start=start, target=target, loss=G.calibration_loss_fn(),
                theta=torch.from_numpy(np.stack(nominal, 1)).requires_grad_(c["grad"]))


def _state(s):
    s["sim"].state_device(s["out"], G.F_ALL, wait=False)
    return s["out"]


def run(state):
    s, sim = state, state["sim"]
    kind = s["kind"]
    if kind in ("ring", "grid", "ensemble", "metro", "jam"):
        if "start" in s:
            sim.write_state(s["start"])
        sim.step(s["steps"])
        return _state(s)
    if kind == "outputs":
        sim.write_state(s["start"])
        sim.step(s["steps"])
        return dict(_state(s), emissions=sim.emissions(), link_times=sim.link_times(), samples=sim.edge_samples())
    if kind == "route":
        sim.route(s["costs"])
        offsets, links = sim.routes()
        s["paths"][:len(links)] = links
        return offsets, s["paths"]
    if kind == "equilibrium":
        cost, gap = sim.equilibrium(SCHEDULE, s["steps"])
        return dict(_state(s), cost=cost, gap=gap)
    if kind == "assign":
        return sim.assign_static(s["capacity"], max_iter=s["iters"])
    theta = s["theta"]
    theta.grad = None
    loss = s["loss"].apply(theta, sim, s["start"], s["target"], s["steps"], s["every"], 64)
    if not s["grad"]:
        return loss
    loss.backward()
    return loss.detach(), theta.grad


# ---------------------------------------------------------------------------- what a pass is
def work(case):
    """Per vehicle-step 40 bytes (position, speed, link, lane, id and route cursor read; position, speed,
    link and lane written) and about 60 operations (Eq. 7, the ballistic update, a share of the lane-change
    evaluations).  Planning: the links with their costs read once and the paths written; one addition and
    one comparison per link and tree."""
    c, kind = case, case["kind"]
    def steps(vehicles, n):
        return dict(bytes=40.0 * vehicles * n, flops=60.0 * vehicles * n)
    if kind == "ring":
        return steps(c["vehicles"], c["steps"])
    if kind == "grid":
        return steps(0.1 * c["hourly"], c["steps"])
    if kind == "ensemble":
        return steps(4500.0 * c["scenarios"], c["steps"])
    if kind == "metro":
        return steps(c["active"], c["steps"])
    if kind == "jam":
        return steps(c["corridors"] * c["lanes"] * math.floor(c["length"] / c["spacing"]), c["steps"])
    if kind == "outputs":
        w = steps(c["active"], c["steps"])
        w["bytes"] += 32.0 * c["active"] * c["steps"]           # the fuel and CO sums, read and written
        return w
    if kind == "calib":
        w = steps(0.06 * c["trips"], c["steps"] * (3 if c["grad"] else 1))
        w["bytes"] += 8.0 * c["trips"] * (c["steps"] // c["every"])   # the target progress
        return w
    nodes = c["nx"] * c["ny"]
    links = 2 * round(275_000 * nodes / 225_000)
    hops = 0.4 * (c["nx"] + c["ny"]) / 2
    trees = nodes * (1 - math.exp(-c["trips"] / nodes))
    plan = dict(bytes=12.0 * links + c["trips"] * (12 + 4 * hops), flops=2.0 * links * trees)
    if kind == "route":
        return plan
    if kind == "assign":
        return dict(bytes=(c["iters"] + 1) * (plan["bytes"] + 40.0 * links), flops=(c["iters"] + 1) * plan["flops"])
    w = steps(0.5 * c["trips"], c["steps"])
    return dict(bytes=4 * (w["bytes"] + plan["bytes"]), flops=4 * w["flops"] + 2.8 * plan["flops"])


def exact(case, seed):
    """The ring in binary64.  The other trajectories, loads and gradients follow discrete decisions
    (admissions, lane changes, tied shortest paths) that the model defines in binary32 and whole
    numbers: no 64-bit run takes the same ones."""
    if case["kind"] != "ring":
        return None
    sc = S.ring(n_veh=case["vehicles"], circumference=20.0 * case["vehicles"], seed=S.BASE_SEED + seed)
    n, L = case["vehicles"], 20.0 * case["vehicles"]
    x, v = sc["init_state"]["x"].astype(np.float64), sc["init_state"]["v"].astype(np.float64)
    v0, T, a, b, s0, dt = 30.0, 1.5, 1.0, 1.5, 2.0, 0.5
    for _ in range(case["steps"]):
        order = np.argsort(x, kind="stable")
        lead = np.empty(n, np.int64)
        lead[order] = np.roll(order, -1)
        gap = np.where(x[lead] > x, x[lead] - x, L - x + x[lead]) - 5.0
        want = s0 + np.maximum(0.0, v * T + v * (v - v[lead]) / (2 * math.sqrt(a * b)))
        acc = a * (1 - (v / v0) ** 4 - (want / np.maximum(gap, 0.1)) ** 2)
        go = v + acc * dt >= 0
        step = np.where(go, v * dt + 0.5 * acc * dt * dt, -(v * v) / np.where(go, 1.0, 2 * acc))
        x, v = x + step, np.where(go, v + acc * dt, 0.0)
        x = np.where(x >= L, x - L, x)
    out = {k: None for k, _ in FIELDS}
    return dict(out, x=x, v=v)
