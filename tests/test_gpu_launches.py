"""The launches of many time steps from the outside: how many a call makes,
what happens once a device-side wait has given up, captured launches, several
contexts at once, and the scan of the medium that precedes them."""
import time

import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def fw2(fw2lib):
    from paper_2106_11476_gb300 import fw2 as m
    return m


FIELDS = ("p", "vx", "vy", "psi1x", "psi1y", "psi2x", "psi2y")


def problem(nx, ny, steps=0, seed=0):
    prob = synth.homogeneous((nx, ny), 1e-4, 0.0, relax=synth.relaxation_sets()["N2_y1.0_a0.5"], beta=4.0)
    prob.c = (1500 + 100 * np.random.default_rng(seed).random(prob.grid_shape)).astype(np.float32)
    prob.nl_mode, prob.dt = "pressure", 0.3 * 1e-4 / 2200.0
    prob.pml_transition, prob.pml_bound = 5, 3
    prob.n_steps = steps
    if steps:
        prob.sensors = synth.Sensors(idx=np.arange(30, dtype=np.int64) * 7, group=np.arange(30, dtype=np.int32) // 10,
                                     n_groups=3)
    return prob


def simulation(fw2, prob, **kw):
    sim = fw2.Simulation(prob, **kw)
    sim.set_state(synth.random_state(prob, seed=9))
    return sim


def assert_same(a, b):
    for f in FIELDS:
        want = b.field(f)
        assert np.isfinite(want).all() and np.abs(want).max() > 0
        np.testing.assert_array_equal(a.field(f), want, err_msg=f)


# ---------------------------------------------------------------- counts ---

@pytest.mark.parametrize("steps,launches", [(1, 2), (2, 2), (256, 2), (257, 4), (519, 5)])
def test_a_call_makes_one_launch_per_256_steps_and_one_per_last_row(fw2, steps, launches):
    """519 steps: 256 + 256 + 7, whose last one has no trace row."""
    prob = problem(64, 40, steps=518)
    sim = simulation(fw2, prob)
    before = sim.launches
    sim.step(steps)
    assert sim.launches - before == launches
    assert fw2.fw2_kernel_path(sim.ctx) == "pipe"
    before = sim.launches
    fw2.fw2_step_part(sim.ctx, 0)
    assert sim.launches - before == 1 and fw2.fw2_kernel_path(sim.ctx) == "pipe"
    sim.close()


# --------------------------------------------------- waits that give up ---

def test_grid_barrier_gives_up_on_a_block_that_never_comes(fw2):
    t0 = time.perf_counter()
    assert fw2.fw2_selftest_grid_barrier(2_000_000) is True               # 2 ms limit
    assert time.perf_counter() - t0 < 5.0
    # the status word of another block's wait ends it before its limit
    t0 = time.perf_counter()
    assert fw2.fw2_selftest_grid_barrier(8_000_000_000, status_set=True) is True
    assert time.perf_counter() - t0 < 4.0
    with pytest.raises(fw2.Fw2Error):
        fw2.fw2_selftest_grid_barrier(0)


def test_after_an_abandoned_wait_nothing_steps_until_a_reset(fw2):
    prob = problem(600, 300)
    sim = simulation(fw2, prob)
    sim.step(5)
    before = {f: sim.field(f) for f in FIELDS}
    fw2.fw2_selftest_abandon(sim.ctx)
    sim.step(4)
    with pytest.raises(fw2.Fw2Error) as e:
        sim.synchronize()
    assert e.value.status == fw2.ETIMEOUT
    for f, want in before.items():
        np.testing.assert_array_equal(sim.field(f), want, err_msg=f)
    fw2.fw2_reset(sim.ctx)
    sim.set_state(synth.random_state(prob, seed=9))
    sim.step(7)
    sim.synchronize()
    fresh = simulation(fw2, prob)
    fresh.step(7)
    assert_same(sim, fresh)
    sim.close()
    fresh.close()


# ------------------------------------------------------ capture, streams ---

def test_captured_launches_replay(fw2):
    """A graph of fw2_step calls replayed three times equals as many steps."""
    import torch
    prob = problem(500, 300)
    stream = torch.cuda.Stream()
    sim, ref = simulation(fw2, prob, stream=stream), simulation(fw2, prob)
    sim.step(3)                        # coefficients and sources are built before the capture
    sim.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream, capture_error_mode="thread_local"):
        sim.step(4)
        sim.step(1)
    for _ in range(3):
        graph.replay()
    torch.cuda.synchronize()
    sim.synchronize()
    ref.step(3 + 3 * 5)
    assert_same(sim, ref)
    sim.close()
    ref.close()


@pytest.mark.parametrize("sizes", [((250, 186),) * 3,                     # side by side on the device
                                   ((600, 500), (520, 300), (250, 186))])  # more blocks than SMs together
def test_contexts_on_streams_of_their_own_step_at_once(fw2, sizes):
    import torch
    probs = [problem(nx, ny, steps=60, seed=i) for i, (nx, ny) in enumerate(sizes)]
    sims = [simulation(fw2, p, stream=torch.cuda.Stream()) for p in probs]
    torch.cuda.synchronize()
    for _ in range(4):
        for s in sims:
            s.step(15)
    for s, p in zip(sims, probs):
        s.synchronize()
        alone = simulation(fw2, p, kernel_path="tile")
        alone.step(60)
        assert_same(s, alone)
        np.testing.assert_array_equal(s.trace.cpu().numpy(), alone.trace.cpu().numpy())
        alone.close()
        s.close()


# ------------------------------------------------------------ medium scan ---

@pytest.mark.parametrize("medium", ["uniform", "random", "huge", "tiny", "mixed"])
def test_medium_scan_finds_the_fp64_maximum(fw2, medium):
    """dt = CFL h / max c / sqrt(kappa1 kappa2): the scan's float pass only
    picks the cells whose quotient is evaluated in FP64, and products beyond
    1e30 or below 1e-30 always are."""
    prob = problem(700, 45)
    rng = np.random.default_rng(1)
    shape = prob.grid_shape
    prob.dt = 0.0
    if medium == "uniform":
        prob.c = np.full(shape, 1540.3, np.float32)
    k1 = (0.8 + 0.4 * rng.random(shape)).astype(np.float32)
    k2 = (0.8 + 0.4 * rng.random(shape)).astype(np.float32)
    if medium == "uniform":
        k1, k2 = np.full(shape, 0.9, np.float32), np.full(shape, 1.1, np.float32)
    some = rng.random(shape) < 0.3
    if medium in ("huge", "mixed"):
        k1[some], k2[some] = 3e20, 2e15
    if medium in ("tiny", "mixed"):
        k1[~some], k2[~some] = k1[~some] * np.float32(1e-20), k2[~some] * np.float32(1e-15)
    prob.kappa1, prob.kappa2 = k1, k2
    sim = fw2.Simulation(prob)
    c = np.asarray(prob.c, np.float64)
    want = 0.4 * prob.h / (c / np.sqrt(k1.astype(np.float64) * k2.astype(np.float64))).max()
    assert abs(sim.dt / want - 1.0) < 1e-14
    sim.close()


def test_medium_scan_counts_the_invalid_cells(fw2):
    prob = problem(700, 45)
    prob.rho = np.full(prob.grid_shape, 1000.0, np.float32)
    prob.c[3, 5], prob.c[44, 699], prob.rho[0, 0], prob.rho[20, 300] = np.nan, -1.0, np.inf, 0.0
    with pytest.raises(fw2.Fw2Error) as e:
        fw2.Simulation(prob)
    assert e.value.status == fw2.EINVAL and "4 cells have" in str(e.value)
