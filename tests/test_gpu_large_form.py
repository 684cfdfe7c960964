"""The step's kernels for large handles (the lane scan and the placement by
slots), reached at small sizes: a handle takes that form by its number of
trips, so trips that never depart within the test are added behind the others.
A vehicle's results depend on its own id and on the vehicles near it only, so
they have to be what the handle without the added trips gives (the placement
by tiles), bit for bit, and what the FP64 oracle gives."""
import dataclasses
import time

import numpy as np
import pytest

import oracle
from handmade import one_road
from paper_2406_10661_gb300 import binding, scenario as sc

pytestmark = pytest.mark.gpu

ADDED = 600_001  # trips that reach the form by themselves
NEVER = 1 << 30


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    binding.load()


def _more(veh, lane=0):
    """The trips and ADDED more on a lane (of road 0) that never depart."""
    off = veh.route_off[-1] + 1 + np.arange(ADDED, dtype=np.int64)
    return sc.Vehicles(n=veh.n + ADDED, route_off=np.concatenate([veh.route_off, off]).astype(np.int32),
                       routes=np.concatenate([veh.routes, np.zeros(ADDED)]).astype(np.int32),
                       start_lane=np.concatenate([veh.start_lane, np.full(ADDED, lane)]).astype(np.int32),
                       dep=np.concatenate([veh.dep, np.full(ADDED, NEVER)]).astype(np.int32),
                       v0f=np.concatenate([veh.v0f, np.ones(ADDED)]).astype(np.float32))


def _large(scen):
    return dataclasses.replace(scen, veh=_more(scen.veh))


def _set(sim, st, n):
    """The state with the vehicles past it (to n of them) waiting."""
    k = n - len(st["status"])
    rest = {"status": 0, "lane": -1, "s": 0, "v": 0, "rc": 0}
    sim.set_state(*(np.concatenate([st[x], np.full(k, rest[x], st[x].dtype)]) for x in rest), 0)


def _pair(scen, precision, st=None):
    large = _large(scen)
    a = binding.Simulation(scen.net, scen.veh, scen.params, precision=precision)
    b = binding.Simulation(large.net, large.veh, large.params, precision=precision)
    assert a.step_launches() == 2 and b.step_launches() == 3
    if st is not None:
        _set(a, st, scen.veh.n); _set(b, st, large.veh.n)
    return a, b


def _same_state(x, y, n):
    for k in ("status", "lane", "rc", "s", "v", "flags"):
        assert np.array_equal(x[k][:n], y[k][:n]), k


def _same(a, b, n, waiting=ADDED):
    _same_state(a.state(), b.state(), n)
    am, bm = a.metrics(), b.metrics()
    bm["n_waiting"] -= waiting
    assert am == bm and am["errors"] == 0


def _as_oracle(sim, ora, n):
    g, r = sim.state(), ora.state()
    act = r["status"] == 1
    assert np.array_equal(g["status"][:n], r["status"]) and np.array_equal(g["flags"][:n], r["flags"])
    for k in ("lane", "rc"):
        assert np.array_equal(g[k][:n][act], r[k][act]), k
    # FP64 on both sides: a step's rounding (1e-16 relative) grows by a few digits over the rollout
    for k in ("s", "v"):
        assert np.abs(g[k][:n][act] - r[k][act]).max(initial=0) < 1e-6, k


@pytest.mark.parametrize("precision", [32, 64])
@pytest.mark.parametrize("n,lanes", [(1, 1), (255, 1), (256, 1), (257, 1), (513, 2), (1800, 1), (2600, 2)])
def test_long_segments(n, lanes, precision):
    """Segments at the edges of a 256-slot tile and over many tiles, every
    vehicle attempting lane changes."""
    rng = np.random.RandomState(n)
    length = 9.0 * -(-n // lanes) + 50.0
    scen, st = one_road(lanes, length, [(k % lanes, length - 1.0 - 9.0 * (k // lanes) - rng.uniform(0, 0.3),
                                         rng.uniform(0.0, 10.0), rng.uniform(0.8, 1.2)) for k in range(n)],
                        params=sc.Params(seed=3, p_attempt=1.0))
    if precision == 32:
        st = {k: v.astype(np.float32).astype(v.dtype) for k, v in st.items()}
    a, b = _pair(scen, precision, st)
    ora = oracle.Oracle(scen.net, scen.veh, scen.params)
    _set(ora, st, n)
    for _ in range(3):
        a.step(9); b.step(9); ora.step(9)
        _same(a, b, n)
        if precision == 64:
            _as_oracle(b, ora, n)


# lanes in all: 1023, 1024, 1025, 2047, 2048, 4094 .. 4099: the remainders of a 4-lane load and of a scan tile
@pytest.mark.parametrize("n_lanes", [1, 1023, 1024, 1025, 2047, 2048, 4094, 4095, 4096, 4097, 4099, 8193])
def test_lane_counts(n_lanes):
    """A corridor of one-lane roads, with a second one to make up the number of
    lanes, as a batch: transfers over the whole scan."""
    parts = [n_lanes] if n_lanes % 2 else [n_lanes - 1, 1]
    scens = []
    for i, k in enumerate(parts):  # k lanes: (k + 1) / 2 roads, the others join them
        roads = (k + 1) // 2
        net = sc.corridor_network(1, (60.0,) * roads)
        cars = np.arange(0, roads, 2)
        veh = sc.Vehicles(n=len(cars), route_off=np.concatenate([[0], np.cumsum(roads - cars)]).astype(np.int32),
                          routes=np.concatenate([np.arange(c, roads) for c in cars]).astype(np.int32),
                          start_lane=cars.astype(np.int32), dep=(cars % 7).astype(np.int32),
                          v0f=np.ones(len(cars), np.float32))
        assert net.n_lanes == k
        scens.append(sc.Scenario(net, veh, sc.Params(scenario=i), f"corridor{k}"))
    a = binding.Batch(scens, precision=64)
    b = binding.Batch([_large(scens[0]), *scens[1:]], precision=64)
    assert b.step_launches() == 3
    for _ in range(3):
        a.step(13); b.step(13)
        for i, s in enumerate(scens):
            _same_state(a.state(i), b.state(i), s.veh.n)
            am, bm = a.metrics(i), b.metrics(i)
            bm["n_waiting"] -= ADDED if i == 0 else 0
            assert am == bm and am["errors"] == 0
    for i, s in enumerate(scens):
        ora = oracle.Oracle(s.net, s.veh, s.params)
        ora.step(39)
        g, r = b.state(i), ora.state()
        assert np.array_equal(g["status"][:s.veh.n], r["status"])
        assert np.array_equal(g["lane"][:s.veh.n], r["lane"])


@pytest.mark.parametrize("precision", [32, 64])
@pytest.mark.parametrize("groups,p_attempt", [(False, 0.3), (True, 0.3), (True, 1.0)])
def test_lane_changes_and_groups(groups, p_attempt, precision):
    """Optional and mandatory changes: many entrants per lane."""
    scen = sc.small_groups_scenario() if groups else sc.small_scenario()
    scen.params.p_attempt = p_attempt
    a, b = _pair(scen, precision)
    ora = oracle.Oracle(scen.net, scen.veh, scen.params)
    for _ in range(3):
        a.step(90); b.step(90); ora.step(90)
        _same(a, b, scen.veh.n)
        if precision == 64:
            _as_oracle(b, ora, scen.veh.n)
    assert b.metrics()["lane_changes"] > 0


def test_max_pressure_and_closures():
    """Adaptive signals (their sums and their phases belong to two kernels of
    the step) and lanes closed and slowed on the way."""
    scen = sc.small_scenario()
    a, b = _pair(scen, 64)
    ora = oracle.Oracle(scen.net, scen.veh, scen.params)
    J = np.arange(scen.net.n_junctions, dtype=np.int32)
    for k in range(4):
        for sim in (a, b):
            if k == 1:
                sim.set_signal_policy(J, binding.POLICY_MAX_PRESSURE)
            if k == 2:
                sim.set_lane_restriction([3, 8], [1, 1]); sim.set_lane_max_speed([5], [6.0])
        if k == 1:
            ora.set_signal(list(J), oracle.POLICY_MAX_PRESSURE)
        a.step(70); b.step(70)
        _same(a, b, scen.veh.n)
        for x, y in zip(a.signal_state(J), b.signal_state(J)):
            assert np.array_equal(x, y)
        if k < 2:
            ora.step(70)
            _as_oracle(b, ora, scen.veh.n)


@pytest.mark.parametrize("precision", [32, 64])
def test_batch(precision):
    """Uneven members, one without vehicles or junctions: each as alone."""
    net = sc.corridor_network(2, (500.0,))
    none = sc.Vehicles(n=0, route_off=np.zeros(1, np.int32), routes=np.zeros(0, np.int32),
                       start_lane=np.zeros(0, np.int32), dep=np.zeros(0, np.int32), v0f=np.zeros(0, np.float32))
    scens = [sc.small_scenario(seed=4), sc.Scenario(net, none, sc.Params(), "empty"), sc.small_groups_scenario(seed=5),
             sc.small_scenario(seed=6)]
    for i, s in enumerate(scens):
        s.params.scenario = i
    batch = binding.Batch([*scens[:3], _large(scens[3])], precision=precision)
    assert batch.step_launches() == 3
    for n in (1, 8, 141):
        batch.step(n)
    for i, s in enumerate(scens):
        alone = binding.Simulation(s.net, s.veh, s.params, precision=precision)
        assert alone.step_launches() == 2
        alone.step(150)
        _same_state(alone.state(), batch.state(i), s.veh.n)
        am, bm = alone.metrics(), batch.metrics(i)
        bm["n_waiting"] -= ADDED if i == 3 else 0
        assert am == bm, i


@pytest.mark.parametrize("precision", [32, 64])
def test_slots_freeze_retire_and_reuse(precision):
    """Slots whose capacity reaches the form: scenarios frozen at horizons
    within and at the end of the steps launched together, retired and replaced
    while others run."""
    scens = [sc.small_scenario(seed=k + 1) for k in range(4)]
    need = [binding.slot_caps(s) for s in scens]
    caps = [{k: max(c[k] for c in need) for k in need[0]} for _ in range(2)]
    caps[1]["n_vehicles"] = ADDED
    slots = binding.Slots(caps, scens[0].params, precision=precision)
    assert slots.step_launches() == 3

    def check(slot, scen, steps):
        alone = binding.Simulation(scen.net, scen.veh, scen.params, precision=precision)
        assert alone.step_launches() == 2
        alone.step(steps)
        assert slots.metrics(slot) == alone.metrics()
        _same_state(alone.state(), slots.state(slot), scen.veh.n)

    slots.load(0, scens[0]); slots.set_horizon(0, 93)
    slots.step(40)
    slots.load(1, scens[1]); slots.set_horizon(1, 80)
    slots.step(80)
    check(0, scens[0], 93)
    check(1, scens[1], 80)
    slots.retire(0)
    slots.step(1)
    slots.load(0, scens[2])
    slots.step(7)
    slots.retire(1)
    slots.step(1)
    slots.load(1, scens[3])
    slots.step(60)
    check(0, scens[2], 68)
    check(1, scens[3], 60)


@pytest.mark.parametrize("precision", [32, 64])
def test_single_launch(precision):
    """The step as one cooperative launch, entered and left on the way."""
    scen = sc.small_groups_scenario()
    a, b = _pair(scen, precision)
    a.step(121)
    b.step(40)
    b.set_step_mode(1)
    b.step(41)
    b.set_step_mode(0)
    b.step(40)
    _same(a, b, scen.veh.n)


def test_scan_tiles_of_several_rounds():
    """A member behind more lanes than the scan has tiles for in single rounds
    (4,194,304): its offsets are carried over the rounds and the tiles."""
    net = sc.corridor_network(100, (60.0,) * 21_600)
    assert net.n_lanes > 4_194_304
    veh = sc.Vehicles(n=1, route_off=np.array([0, 1], np.int32), routes=np.array([21_599], np.int32),
                      start_lane=np.array([2_159_999], np.int32), dep=np.array([3], np.int32), v0f=np.ones(1, np.float32))
    scens = [sc.Scenario(net, veh, sc.Params(), "long"), sc.small_groups_scenario()]
    scens[1].params.scenario = 1
    batch = binding.Batch([scens[0], _large(scens[1])], precision=64)
    assert batch.step_launches() == 3
    alone = binding.Simulation(scens[1].net, scens[1].veh, scens[1].params, precision=64)
    for n in (5, 75):
        batch.step(n); alone.step(n)
        _same_state(alone.state(), batch.state(1), scens[1].veh.n)
    assert batch.state(0)["status"][0] == 2 and batch.metrics(0)["errors"] == 0


def test_scan_of_spare_lanes_is_bound_by_memory():
    """The scan of a pool with 1.6 million lanes, most of them spare, from cold
    caches: within three times its 24 bytes per lane at 6.8 TB/s, and 5 us for
    the launch and the events."""
    import torch
    scen = sc.small_scenario()
    caps = dict(binding.slot_caps(scen), n_lanes=1_600_000, n_vehicles=ADDED)
    slots = binding.Slots([caps], scen.params)
    slots.load(0, scen)
    slots.step(60)
    cold = torch.empty(1 << 28, dtype=torch.uint8, device="cuda")
    us = []
    for _ in range(20):
        cold.add_(1)
        torch.cuda.synchronize()
        slots.set_kernel_timing(True)
        slots.step(1)
        slots.synchronize()
        ms, steps = slots.kernel_times()
        us.append(1e3 * ms["lanescan"] / steps)
    slots.set_kernel_timing(False)
    assert np.median(us) < 3 * 24 * 1.6e6 / 6.8e6 + 5, us


def test_a_burst_of_lane_changes_counts_little():
    """The first step of a state in which many vehicles have to change lanes at
    once: k_decide takes no longer with the few tiles of the scan than with the
    many of the placement by tiles (a quarter for the events' 2 us and the clocks)."""
    net = sc.grid_network(30, 300.0, 3, 13.89, lane_groups=True)
    n = 70_000
    rng = np.random.RandomState(1)
    # along every lane, each with a turn drawn among those of its road
    lane = np.sort(rng.randint(0, net.n_road_lanes, n)).astype(np.int32)
    first = np.concatenate([[0], np.flatnonzero(np.diff(lane)) + 1])
    rank = np.arange(n) - np.repeat(first, np.diff(np.append(first, n)))
    s = 285.0 - 30.0 * rank - rng.uniform(0.0, 24.0, n)
    keep = s > 1.0
    lane, s = lane[keep], s[keep]
    road = net.lane_road()
    turn = net.jl_off - net.n_road_lanes
    follow = [np.unique(road[net.jl_target[turn[a]:turn[b]]]) for a, b in
              zip(net.road_lane_off[:-1], net.road_lane_off[1:])]
    go = np.array([follow[r][rng.randint(len(follow[r]))] for r in road[lane]])
    n = len(lane)
    veh = sc.Vehicles(n=n, route_off=(2 * np.arange(n + 1)).astype(np.int32),
                      routes=np.stack([road[lane], go], 1).ravel().astype(np.int32), start_lane=lane,
                      dep=np.zeros(n, np.int32), v0f=np.ones(n, np.float32))
    st = {"status": np.ones(n, np.int32), "lane": lane, "s": s, "v": np.full(n, 2.0), "rc": np.zeros(n, np.int32)}
    a = binding.Simulation(net, veh, sc.Params(p_attempt=1.0))
    b = binding.Simulation(net, _more(veh), sc.Params(p_attempt=1.0))
    assert b.step_launches() == 3
    us = {}
    for sim, total in ((a, n), (b, n + ADDED)):
        x = []
        for _ in range(15):
            _set(sim, st, total)
            sim.set_kernel_timing(True)
            sim.step(1)
            sim.synchronize()
            x.append(1e3 * sim.kernel_times()[0]["decide"])
            sim.set_kernel_timing(False)
        us[total] = np.median(x)
    assert a.metrics()["lane_changes"] > 15 * n // 10  # (15 steps of at least n / 10)
    _same(a, b, n)
    assert us[n + ADDED] < 1.25 * us[n], us


def test_single_launch_keeps_the_form():
    """The step as one launch scans and places by slots in a large handle too:
    2,464,950 vehicles on the road take at most 1.3 times the three kernels
    (the barriers and the lower occupancy; by tiles 1.4 times and more)."""
    scen, (status, lane, s, v, rc) = sc.saturated_city()
    sim = binding.Simulation(scen.net, scen.veh, scen.params)
    sim.set_state(status, lane, s, v, rc, 0)
    sim.step(8)
    us = {}
    for mode in (0, 1):
        sim.set_step_mode(mode)
        sim.step(8)
        x = []
        for _ in range(7):
            sim.synchronize()
            t = time.perf_counter()
            sim.step(16)
            sim.synchronize()
            x.append((time.perf_counter() - t) / 16e-6)
        us[mode] = np.median(x)
    assert us[1] < 1.3 * us[0], us


@pytest.mark.parametrize("lanescan,lanes_per_thread", [(1, 8), (1, 16), (32, 8), (32, 16)])
@pytest.mark.parametrize("roads", [1023, 1025, 4097, 160_000])
def test_scan_schedules(roads, lanescan, lanes_per_thread):
    """The scan's blocks per SM and lanes per thread, as documented: every
    choice gives the same result, with fewer blocks than tiles too, and from
    one step to the next."""
    net = sc.corridor_network(1, (60.0,) * roads)
    at = np.linspace(0, roads - 1, 500).astype(np.int64)
    veh = sc.Vehicles(n=500, route_off=np.concatenate([[0], np.cumsum(np.minimum(roads - at, 9))]).astype(np.int32),
                      routes=np.concatenate([np.arange(x, min(x + 9, roads)) for x in at]).astype(np.int32),
                      start_lane=at.astype(np.int32), dep=(np.arange(500) % 5).astype(np.int32),
                      v0f=np.ones(500, np.float32))
    a = binding.Simulation(net, _more(veh), sc.Params())
    b = binding.Simulation(net, _more(veh), sc.Params())
    assert b.step_launches() == 3
    a.step(33)
    b.step(7)
    default = b.schedule()
    sched = dict(default, lanescan=lanescan, lanes_per_thread=lanes_per_thread)
    b.set_schedule(**sched)
    assert b.schedule() == sched
    b.step(17)
    b.set_schedule(**default)
    b.step(9)
    _same(a, b, 500, waiting=0)
    assert a.metrics()["n_arrived"] + a.metrics()["n_active"] == 500


@pytest.mark.parametrize("side,trips,launches", [(4, 1000, 2), (12, 12007, 2), (30, 15000, 2), (30, 100_000, 2),
                                                 (60, 20_000, 2), (100, 1000, 3)])
def test_form_follows_vehicles_and_lanes(side, trips, launches):
    """The form whose step was measured faster: three-lane grids, by trips and
    by lanes (471,624 at the last), and the same results with many lanes."""
    net = sc.grid_network(side, 200.0, 3, 13.89)
    veh = sc.random_demand(net, trips, 60, seed=1, dest_pool=64)
    sim = binding.Simulation(net, veh, sc.Params())
    assert sim.step_launches() == launches
    if side == 60:  # (tiles of 256 lanes)
        large = binding.Simulation(net, _more(veh), sc.Params())
        sim.step(90); large.step(90)
        _same(sim, large, trips)


@pytest.mark.parametrize("precision", [32, 64])
@pytest.mark.parametrize("past", [0, 1])
def test_both_sides_of_the_line(past, precision):
    """The heaviest handle that takes the placement by tiles and the next one:
    the same rollout, FP64 as the oracle's."""
    scen = sc.small_scenario()
    k = (1_200_000 - 4 * scen.net.n_lanes) // 2 + past
    veh = _more(scen.veh)
    end = int(veh.route_off[k])
    veh = sc.Vehicles(n=k, route_off=veh.route_off[:k + 1], routes=veh.routes[:end], start_lane=veh.start_lane[:k],
                      dep=veh.dep[:k], v0f=veh.v0f[:k])
    sim = binding.Simulation(scen.net, veh, scen.params, precision=precision)
    assert sim.step_launches() == 2 + past
    a = binding.Simulation(scen.net, scen.veh, scen.params, precision=precision)
    sim.step(150); a.step(150)
    _same(a, sim, scen.veh.n, waiting=k - scen.veh.n)
    if precision == 64:
        ora = oracle.Oracle(scen.net, scen.veh, scen.params)
        ora.step(150)
        _as_oracle(sim, ora, scen.veh.n)
