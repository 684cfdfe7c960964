"""The tiles of the place kernel and the runs of the decision kernel at their
edges, against the FP64 oracle: lanes much longer than a tile, segments at
multiples of the tile, roads with more vehicles than a block has threads, and
many vehicles that enter one lane in one step."""
import numpy as np
import pytest

import oracle
import test_gpu_large_form as large
from paper_2406_10661_gb300 import binding, scenario as sc

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    binding.load()


def _line(n, lanes, spacing, seed=0):
    """n vehicles one behind the other on the first of two roads."""
    rng = np.random.RandomState(seed)
    per_lane = -(-n // lanes)
    net = sc.corridor_network(lanes, (per_lane * spacing + 50.0, 400.0))
    lane = np.arange(n) % lanes
    veh = sc.corridor_vehicles(net, lane, np.zeros(n), v0f=rng.uniform(0.8, 1.2, n))
    s = net.lane_length[0].astype(np.float64) - 1.0 - spacing * (np.arange(n) // lanes) - rng.uniform(0, 0.3, n)
    v = rng.uniform(0.0, 10.0, n)
    return net, veh, {"status": np.ones(n, np.int32), "lane": lane.astype(np.int32), "s": s, "v": v,
                      "rc": np.zeros(n, np.int32)}


def _check(sim, ora):
    g, r = sim.state(), ora.state()
    act = r["status"] == 1
    assert np.array_equal(g["status"], r["status"])
    for k in ("lane", "rc"):
        assert np.array_equal(g[k][act], r[k][act]), k
    assert np.array_equal(g["flags"], r["flags"])
    # FP64 on both sides: the rounding of a step (1e-16 relative) grows over 40 steps by a few digits at most
    for k in ("s", "v"):
        assert np.abs(g[k][act] - r[k][act]).max(initial=0) < 1e-6, k
    gm, rm = sim.metrics(), ora.metrics()
    for k in ("n_active", "n_arrived", "lane_changes", "flagged", "overlaps", "inserted", "mobil_evals", "errors"):
        assert gm[k] == rm[k], (k, gm[k], rm[k])


# 255..257, 511..513: segments at a tile's and a pass's edge; 4095..4097 and 5000: more slot rounds than are held at once
@pytest.mark.parametrize("n,lanes", [(1, 1), (255, 1), (256, 1), (257, 1), (511, 2), (513, 3), (4095, 1), (4097, 1),
                                     (5000, 1), (5000, 3)])
def test_long_segments(n, lanes):
    net, veh, st = _line(n, lanes, 9.0)
    sim = binding.Simulation(net, veh, sc.Params(seed=3), precision=64)
    ora = oracle.Oracle(net, veh, sc.Params(seed=3))
    for o in (sim, ora):
        o.set_state(st["status"], st["lane"], st["s"], st["v"], st["rc"], 0)
    for _ in range(4):
        sim.step(10); ora.step(10)
        _check(sim, ora)


@pytest.mark.parametrize("lanescan,lanes_per_thread", [(1, 16), (1, 8), (32, 16)])
def test_tile_sizes(lanescan, lanes_per_thread):
    """Lane weights and tile sizes from the smallest to the largest give one result."""
    net, veh, st = _line(1500, 3, 8.5)
    sim = binding.Simulation(net, veh, sc.Params(seed=5), precision=64)
    ora = oracle.Oracle(net, veh, sc.Params(seed=5))
    for o in (sim, ora):
        o.set_state(st["status"], st["lane"], st["s"], st["v"], st["rc"], 0)
    sim.step(7); ora.step(7)
    sim.set_schedule(lanescan=lanescan, lanes_per_thread=lanes_per_thread)
    sim.step(23); ora.step(23)
    _check(sim, ora)


@pytest.mark.parametrize("precision", [32, 64])
@pytest.mark.parametrize("p_attempt", [0.0, 0.3, 1.0])
def test_attempt_draw(precision, p_attempt):
    """The attempt draw at its ends: MOBIL evaluations as the oracle counts them in one step."""
    net, veh, st = _line(700, 3, 12.0)
    if precision == 32:
        st["s"] = st["s"].astype(np.float32).astype(np.float64)
        st["v"] = st["v"].astype(np.float32).astype(np.float64)
    prm = sc.Params(seed=11, p_attempt=p_attempt)
    sim = binding.Simulation(net, veh, prm, precision=precision)
    ora = oracle.Oracle(net, veh, prm)
    for o in (sim, ora):
        o.set_state(st["status"], st["lane"], st["s"], st["v"], st["rc"], 4)
        o.step(1)
    assert sim.metrics()["mobil_evals"] == ora.metrics()["mobil_evals"]
    assert (p_attempt > 0) == (sim.metrics()["mobil_evals"] > 0)


# 40 .. 520 entrants of one lane in one step: some held in shared memory (up to 128 per tile), some listed, and the
# tiles' lanes mixed; (1, 40): the lanes of a whole tile with one or two each
@pytest.mark.parametrize("precision", [32, 64])
@pytest.mark.parametrize("n,lanes", [(40, 2), (127, 2), (128, 2), (129, 2), (257, 3), (520, 2), (1040, 4)])
def test_many_entrants_of_a_lane(n, lanes, precision):
    """Everyone attempts a change and gains by any: bursts from the full lane into the others, each step."""
    rng = np.random.RandomState(n)
    net = sc.corridor_network(lanes, (14.0 * n + 100.0, 400.0))
    lane = np.full(n, lanes - 1)
    lane[::5] = rng.randint(0, lanes, len(lane[::5]))
    s = net.lane_length[0].astype(np.float64) - 20.0 - 14.0 * np.arange(n) - rng.uniform(0, 2.0, n)
    veh = sc.corridor_vehicles(net, lane, np.zeros(n), v0f=rng.uniform(0.8, 1.2, n))
    st = {"status": np.ones(n, np.int32), "lane": lane.astype(np.int32), "s": s, "v": rng.uniform(4.0, 12.0, n),
          "rc": np.zeros(n, np.int32)}
    if precision == 32:
        st["s"] = st["s"].astype(np.float32).astype(np.float64)
        st["v"] = st["v"].astype(np.float32).astype(np.float64)
    prm = sc.Params(seed=7, p_attempt=1.0, a_th=-3.0)
    sim = binding.Simulation(net, veh, prm, precision=precision)
    assert sim.step_launches() == 2
    ora = oracle.Oracle(net, veh, prm)
    for o in (sim, ora):
        o.set_state(st["status"], st["lane"], st["s"], st["v"], st["rc"], 0)
    if precision == 32:  # (against the placement by slots, bit for bit)
        other = binding.Simulation(net, large._more(veh), prm)
        assert other.step_launches() == 3
        large._set(other, st, n + large.ADDED)
        for _ in range(12):
            sim.step(1); other.step(1)
            large._same(sim, other, n)
        return
    for _ in range(12):
        sim.step(1); ora.step(1)
        _check(sim, ora)
    assert sim.metrics()["lane_changes"] > n // 4


def test_flowing_city_does_not_wait_for_entrants():
    """Some lane of a city in flowing traffic takes several entrants in every step: the placement, at 0.47 of the
    decision's time (0.80 with a lane's entrants one after the other), stays below 0.62 of it."""
    from perf import cases
    sim = cases.prepare({"kind": "sim", "net": "city", "side": 30, "lanes": 3, "length": 300.0, "trips": 50000,
                         "steps": 10, "read": "observe", "precision": 32, "groups": False, "policy": "fixed"}, 7)["sim"]
    assert sim.step_launches() == 2
    sim.step(2000)
    share = []
    for _ in range(9):
        sim.set_kernel_timing(True)
        sim.step(16)
        sim.synchronize()
        ms, _ = sim.kernel_times()
        share.append(ms["place"] / ms["decide"])
        sim.set_kernel_timing(False)
    assert np.median(share) < 0.62, share
