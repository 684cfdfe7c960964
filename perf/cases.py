"""Performance cases: the work that a user of the simulator has it do, through
the public binding (``Simulation``, ``Batch``, ``Slots`` and the allocation-free
lane-offset scan).

A pass of a simulation case is what an optimisation loop does between two of
its decisions: set signal phases (when the case has actions), advance some
steps, read back what the agent looks at.  ``read`` says what that is:

* ``observe``: the queue of every lane, the mean speed of every road and the
  cumulative metrics (a signal agent's observation and reward);
* ``state``: every vehicle's status, lane, position, speed, route cursor and
  flags (trajectory logging, checkpoints).

Passes follow one another on one simulation, so the traffic has to stay what
it is: trips are random walks over the road graph, long enough that about as
many vehicles arrive as depart over ``horizon`` steps (a vehicle needs about a
minute per road, half of it at a red light).
"""
import functools
import math

import numpy as np
import torch

from paper_2406_10661_gb300 import binding, scenario as sc

MINUTE_PER_ROAD = 60.0
METRICS = ("step", "n_active", "n_waiting", "n_arrived", "vehicle_updates", "lane_changes", "flagged", "overlaps",
           "inserted", "errors", "mobil_evals")
METRIC_SUMS = ("tt_sum", "speed_sum")


def _horizon(trips):
    """Steps over which a state stays in balance: small simulations run many
    more steps in the same time."""
    return int(min(30000, max(4000, 1.2e9 / trips)))


def _sim(name, net, side, trips, steps, read, precision=32, lanes=3, length=300.0, groups=False, policy="fixed"):
    return {"name": name, "kind": "sim", "net": net, "side": side, "lanes": lanes, "length": length, "trips": trips,
            "steps": steps, "read": read, "precision": precision, "groups": groups, "policy": policy}


def listed():
    return [
        # the 4x4 workload under closed-loop control: an action and an observation every step, all latency
        _sim("grid4-closed-loop", "grid", 4, 1000, 1, "observe", lanes=2, length=200.0, policy="manual"),
        # 4x4 with turn lanes in FP64, a minute at a time, trajectories kept: validation against double precision
        _sim("grid4-groups-fp64", "grid", 4, 1501, 60, "state", precision=64, length=200.0, groups=True),
        # a small town under adaptive signals: the max-pressure policy compared with learned ones
        _sim("grid12-max-pressure", "grid", 12, 12007, 10, "observe", policy="maxp"),
        # the 30x30 workload as an agent drives it: phases of all 900 junctions every 10 steps
        _sim("grid30-control", "grid", 30, 100000, 10, "observe", policy="manual"),
        # the same in FP64: the precision used to compare trajectories
        _sim("grid30-fp64", "grid", 30, 100000, 10, "observe", precision=64),
        # turn lanes with mandatory changes, two-minute rollouts without interference
        _sim("grid30-groups-rollout", "grid", 30, 99991, 120, "observe", groups=True),
        # a district with every vehicle's trajectory logged each 10 s
        _sim("city45-trajectories", "city", 45, 500009, 10, "state"),
        # the city of 39,600 roads and 2,464,950 trips
        _sim("city100-rollout", "city", 100, 2464950, 10, "observe"),
        # many rollouts of uneven size side by side: one population of a black-box search
        {"name": "batch64-uneven", "kind": "batch", "scenarios": 64, "trips_lo": 2000, "trips_hi": 100000, "steps": 30},
        # rollout requests in the slots of a resident batch, each with its agent
        {"name": "served-slots", "kind": "served", "scenarios": 12, "trips_lo": 5000, "trips_hi": 100000, "steps": 10},
        # lane segments inside another framework's pipeline: the city's lanes, and the largest networks
        {"name": "offsets-city", "kind": "offsets", "lanes": 362353},
        {"name": "offsets-largest", "kind": "offsets", "lanes": 4000003},
    ]


def draw(rng):
    def log(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(("sim", "sim", "sim", "sim", "batch", "served", "offsets"))
    if kind == "offsets":
        return {"kind": kind, "lanes": log(300, 4000003)}
    if kind in ("batch", "served"):
        return {"kind": kind, "scenarios": rng.randint(2, 64 if kind == "batch" else 12), "trips_lo": log(1500, 5000),
                "trips_hi": log(6000, 60000), "steps": rng.choice((10, 30))}
    trips = log(600, 600000)
    net = rng.choice(("grid", "city"))
    lanes, length = rng.randint(1, 4), rng.choice((150.0, 200.0, 300.0))
    # the side at which a trip has 25 to 60 m of lane
    room = trips * rng.uniform(25.0, 60.0)
    per_link = 2 * lanes * length if net == "grid" else 2 * 2.3 * 270.0
    side = max(3, min(100, int(round(math.sqrt(room / per_link / 2)))))
    steps = rng.choice((1, 5, 10, 30)) if trips > 20000 else rng.choice((1, 10, 60))
    return {k: v for k, v in _sim("", net, side, trips, steps, rng.choice(("observe", "observe", "state")),
                                  rng.choice((32, 32, 64)), lanes, length, lanes > 1 and rng.random() < 0.25,
                                  rng.choice(("fixed", "manual", "maxp"))).items() if k != "name"}


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
@functools.lru_cache(maxsize=160)
def _network(net, side, lanes, length, groups, seed):
    """A road network (a user's program keeps it) and its turns: the roads
    that follow a road, padded to the widest junction, and how many they are."""
    if net == "city":
        g = sc.perturbed_grid_network(side, seed=seed, lane_groups=groups)
    else:
        g = sc.grid_network(side, length, lanes, vmax_choices=(11.1, 13.89, 16.67), offsets=True, seed=seed,
                            lane_groups=groups)
    road = g.lane_road()
    turns = np.unique(np.stack([np.repeat(road[:g.n_road_lanes], np.diff(g.jl_off)), road[g.jl_target]], axis=1), axis=0)
    count = np.bincount(turns[:, 0], minlength=g.n_roads)
    table = np.zeros((g.n_roads, int(count.max())), dtype=np.int64)
    table[turns[:, 0], np.arange(len(turns)) - np.repeat(np.cumsum(count) - count, count)] = turns[:, 1]
    return g, table, count


def _trips(network, trips, horizon, seed, depart_within=None):
    """Trips with random-walk routes, and the state in which 70% of them are
    on the road, spread over the lanes with uneven gaps, while the others
    depart over the horizon.  With ``depart_within`` the first 70% depart
    within that many steps instead of being on the road already."""
    net, table, count = network
    dev = "cuda"
    rng = torch.Generator(device=dev).manual_seed(seed)

    def uniform(*shape):
        return torch.rand(*shape, generator=rng, device=dev, dtype=torch.float64)

    table, count = torch.from_numpy(table).to(dev), torch.from_numpy(count).to(dev)
    lane_off = torch.from_numpy(net.road_lane_off.astype(np.int64)).to(dev)
    length = torch.from_numpy(net.lane_length[:net.n_road_lanes].astype(np.float64)).to(dev)
    vmax = torch.from_numpy(net.lane_vmax[:net.n_road_lanes].astype(np.float64)).to(dev)
    lane_road = torch.from_numpy(net.lane_road()[:net.n_road_lanes].astype(np.int64)).to(dev)
    active = int(0.7 * trips)
    # vehicles one behind the other along all lanes, in random order of their ids
    total = length.cumsum(0)
    x = (torch.arange(active, device=dev) + 0.6 * uniform(active)) * (total[-1] / active)
    lane = torch.searchsorted(total, x, right=True).clamp_(max=net.n_road_lanes - 1)
    s = (x - (total - length)[lane]).clamp_(min=0.0).minimum(length[lane])
    v0f = (1.0 + 0.1 * torch.randn(trips, generator=rng, device=dev, dtype=torch.float64)).clamp_(0.7, 1.3)
    ahead = torch.cat([x[1:] - x[:-1], x.new_full((1,), 1e3)])
    ids = torch.randperm(trips, generator=rng, device=dev)
    on, off = ids[:active], ids[active:]
    v = ((ahead - 7.0) / 1.5).clamp_(min=0.0).minimum(v0f[on] * vmax[lane])
    start = (uniform(trips) * net.n_road_lanes).long()
    start[on] = lane
    dep = 1 + (uniform(trips) * (horizon - 1)).long()
    dep[on] = 0 if depart_within is None else (uniform(active) * depart_within).long()
    # routes of 1 to `hops` roads
    hops = max(2, int(horizon / 25))
    lens = 1 + (uniform(trips) * hops).long()
    routes = torch.empty(trips, hops, dtype=torch.int32, device=dev)
    road = lane_road[start]
    for h in range(hops):
        routes[:, h] = road
        road = table[road, (uniform(trips) * count[road]).long()]
    routes = routes[torch.arange(hops, device=dev)[None, :] < lens[:, None]]
    route_off = torch.cat([lens.new_zeros(1), lens.cumsum(0)]).int()
    veh = sc.Vehicles(n=trips, route_off=route_off.cpu().numpy(), routes=routes.cpu().numpy(),
                      start_lane=start.int().cpu().numpy(), dep=dep.int().cpu().numpy(), v0f=v0f.float().cpu().numpy())

    def by_id(value, rest, dtype):
        out = torch.full((trips,), rest, dtype=dtype, device=dev)
        out[on] = value.to(dtype) if isinstance(value, torch.Tensor) else value
        return out.cpu().numpy()

    state = {"status": by_id(1, 0, torch.int32), "lane": by_id(lane, -1, torch.int32),
             "s": by_id(s.float(), 0, torch.float64), "v": by_id(v.float(), 0, torch.float64),
             "rc": np.zeros(trips, dtype=np.int32)}
    return veh, state


def _phases(net, seed, n=8):
    """An agent's actions: n phase settings of all junctions, used in turn."""
    r = np.random.RandomState(seed % (1 << 31))
    return [r.randint(0, 4, net.n_junctions).astype(np.int32) for _ in range(n)]


def _sizes(case):
    """Trips and grid side of the scenarios of a batch, log-uniform, as uneven
    as the range is (their order is fixed: it belongs to the case)."""
    k = case["scenarios"]
    lo, hi = math.log(case["trips_lo"]), math.log(case["trips_hi"])
    out = []
    for i in range(k):
        n = int(round(math.exp(lo + (hi - lo) * ((i * 37 + 11) % k + 0.5) / k)))
        out.append((n, max(5, min(40, int(round(5 * 8 ** (math.log(n / 2000.0) / math.log(150.0))))))))
    return out


def prepare(case, seed):
    kind = case["kind"]
    if kind == "offsets":
        n = case["lanes"]
        rng = torch.Generator(device="cuda").manual_seed(seed)

        def draw_int(hi):
            return torch.randint(0, hi, (n,), generator=rng, device="cuda", dtype=torch.int32)

        # a few vehicles per lane, some of which leave; a few enter
        size = draw_int(12)
        leave = torch.minimum(size, draw_int(3))
        off = torch.cat([size.new_zeros(1), size.cumsum(0).int()])
        out = [torch.empty(n + 1, dtype=torch.int32, device="cuda"), torch.empty(n, dtype=torch.int32, device="cuda")]
        return {"kind": kind, "n": n, "args": [off, leave, draw_int(3)], "out": out}
    if kind == "sim":
        network = _network(case["net"], case["side"], case["lanes"], case["length"], case["groups"], 0)
        net = network[0]
        veh, st = _trips(network, case["trips"], _horizon(case["trips"]), seed)
        sim = binding.Simulation(net, veh, sc.Params(seed=seed), precision=case["precision"])
        sim.set_state(st["status"], st["lane"], st["s"], st["v"], st["rc"], 0)
        junctions = np.arange(net.n_junctions, dtype=np.int32)
        if case["policy"] == "maxp":
            sim.set_signal_policy(junctions, binding.POLICY_MAX_PRESSURE)
        acts = _phases(net, seed) if case["policy"] == "manual" else None
        sim.step(2)  # the launches are loaded
        sim.synchronize()
        return {"kind": kind, "sim": sim, "steps": case["steps"], "read": case["read"], "junctions": junctions,
                "acts": acts, "pass": 0}
    # batches start with every trip waiting; two minutes fill the roads
    sizes = _sizes(case)
    horizon = _horizon(sum(n for n, _ in sizes))
    scens = []
    for i, (n, side) in enumerate(sizes):
        network = _network("grid", side, 3, 300.0, False, i)
        veh, _ = _trips(network, n, horizon, seed * 1000 + i, depart_within=60)
        scens.append(sc.Scenario(network[0], veh, sc.Params(seed=seed * 1000 + i, scenario=i)))
    state = {"kind": kind, "steps": case["steps"], "k": len(scens), "pass": 0}
    if kind == "batch":
        state["sim"] = binding.Batch(scens)
    else:
        state["sim"] = binding.Slots([binding.slot_caps(s) for s in scens], scens[0].params)
        for i, s in enumerate(scens):
            state["sim"].load(i, s)
        nj = [s.net.n_junctions for s in scens]
        state["slots"] = np.concatenate([np.full(n, i, dtype=np.int32) for i, n in enumerate(nj)])
        state["junctions"] = np.concatenate([np.arange(n, dtype=np.int32) for n in nj])
        each = [_phases(s.net, seed + i) for i, s in enumerate(scens)]
        state["acts"] = [np.concatenate(a) for a in zip(*each)]
    state["sim"].step(120)
    state["sim"].synchronize()
    return state


def _metrics(records):
    return {"counts": np.array([[m[k] for k in METRICS] for m in records], dtype=np.int64),
            "sums": np.array([[m[k] for k in METRIC_SUMS] for m in records], dtype=np.float64)}


def _all_metrics(sim, k):
    for i in range(k):
        sim.metrics_enqueue(i, scenario=i)
    return _metrics([sim.metrics_read(i) for i in range(k)])


def run(state):
    kind = state["kind"]
    if kind == "offsets":
        ptrs = [t.data_ptr() for t in state["args"] + state["out"]]
        rc = binding.moss_lane_offsets_noalloc(state["n"], *ptrs, stream=torch.cuda.current_stream().cuda_stream)
        if rc != binding.MOSS_OK:
            raise binding.MossError(rc, "moss_lane_offsets_noalloc")
        return state["out"]
    sim = state["sim"]
    state["pass"] += 1
    if kind == "sim":
        if state["acts"] is not None:
            sim.set_signal_phase(state["junctions"], state["acts"][state["pass"] % len(state["acts"])])
        sim.step(state["steps"])
        if state["read"] == "state":
            return sim.state()
        return {"queue": sim.lane_queue(), "speed": sim.road_speed(), **_metrics([sim.metrics()])}
    if kind == "batch":
        sim.step(state["steps"])
        return _all_metrics(sim, state["k"])
    sim.set_signal_phases(state["slots"], state["junctions"], state["acts"][state["pass"] % len(state["acts"])])
    sim.step(state["steps"])
    return {"queue": [sim.lane_queue(i) for i in range(state["k"])], **_all_metrics(sim, state["k"])}


# ---------------------------------------------------------------------------
def work(case):
    """Bytes and operations of one pass.  A step reads and writes each active
    vehicle's record (position, speed, id, lane, desired-speed factor, route
    cursor, last road, next lane) and reads its lane's record once; reading
    back writes each value once.  About 120 floating-point operations per
    vehicle and step (car following on the own lane, the lane-change
    utilities of every other vehicle, the update)."""
    if case["kind"] == "offsets":
        return {"bytes": 20 * case["lanes"], "flops": 6 * case["lanes"]}
    if case["kind"] == "sim":
        net = _network(case["net"], case["side"], case["lanes"], case["length"], case["groups"], 0)[0]
        active, lanes = int(0.7 * case["trips"]), net.n_lanes
        record = 32 if case["precision"] == 32 else 48
        back = 32 * case["trips"] if case["read"] == "state" else 4 * lanes + 8 * net.n_roads
    else:
        nets = [_network("grid", side, 3, 300.0, False, i)[0] for i, (_, side) in enumerate(_sizes(case))]
        active, lanes, record = int(0.7 * sum(n for n, _ in _sizes(case))), sum(n.n_lanes for n in nets), 32
        back = 4 * lanes if case["kind"] == "served" else 104 * len(nets)
    return {"bytes": case["steps"] * (2 * record * active + 32 * lanes) + back, "flops": case["steps"] * 120 * active}


def exact(case, seed):
    """The lane segments are whole numbers and plain sums.  A simulation has
    no such value: each step takes discrete decisions from its own rounded
    state, and a path that rounds otherwise is another trajectory."""
    if case["kind"] != "offsets":
        return None
    st = prepare(case, seed)
    off, leave, enter = [t.cpu().numpy().astype(np.int64) for t in st["args"]]
    size = np.diff(off) - leave + enter
    return [np.concatenate([[0], np.cumsum(size)]).astype(np.int32),
            np.concatenate([[0], np.cumsum(leave)[:-1]]).astype(np.int32)]
