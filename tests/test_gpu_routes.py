"""Calls that the pipelined 2D path hands to kernels of their own, and launches
that it does not make: the same bits as the tile kernels either way, and the
route that the rule of the sizes says (counted in launches)."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def fw2(fw2lib):
    from paper_2106_11476_gb300 import fw2 as m
    return m


def problem(nx, ny, N=2, steps=6):
    prob = synth.homogeneous((nx, ny), 1e-4, 0.0, relax=synth.relaxation_sets()["N2_y1.0_a0.5"] if N else None, beta=4.0)
    prob.c = (1500 + 100 * np.random.default_rng(3).random(prob.grid_shape)).astype(np.float32)
    prob.nl_mode = "pressure"
    prob.dt = 0.3 * 1e-4 / 2200.0
    if N:
        prob.pml_transition, prob.pml_bound = 5, 3
    prob.n_steps = steps
    prob.sensors = synth.Sensors(idx=np.arange(40, dtype=np.int64) * 5, group=np.zeros(40, np.int32), n_groups=1)
    return prob


def run(fw2, prob, steps, path):
    """Fields, trace and the launches of one fw2_step call."""
    sim = fw2.Simulation(prob, kernel_path=path)
    sim.set_state(synth.random_state(prob, seed=4))
    before = sim.launches
    sim.step(steps)
    n = sim.launches - before
    sim.synchronize()
    assert fw2.fw2_kernel_path(sim.ctx) == ("tile" if path == "tile" else "pipe")
    out = {f: sim.field(f) for f in ("p", "vx", "vy") + (("psi1x", "psi2y") if prob.nrelax else ())}
    out["trace"] = sim.trace.cpu().numpy()
    sim.close()
    return out, n


def same(fw2, prob, steps):
    want, _ = run(fw2, prob, steps, "tile")
    got, launches = run(fw2, prob, steps, "auto")
    assert np.isfinite(want["p"]).all()
    for f, w in want.items():
        np.testing.assert_array_equal(got[f], w, err_msg=f)
    return launches


def sources(idx, group, rows, n_groups):
    sig = np.random.default_rng(5).standard_normal((rows, n_groups)).astype(np.float32)
    return [synth.Source("p", idx, group, 1e3 * sig), synth.Source("vy", idx[:7], group[:7], 1e-3 * sig)]


@pytest.mark.parametrize("nx,ny,cells,repeat,apart", [
    (600, 500, 600 * 500, 1, True),      # every cell
    (600, 500, 2000, 1, False), (203, 77, 203 * 77, 1, False),
    (203, 77, 5, 900, True)])            # 900 entries in each of five cells
def test_dense_and_chained_sources_run_as_kernels_of_their_own(fw2, nx, ny, cells, repeat, apart):
    prob = problem(nx, ny)
    idx = np.tile(np.random.default_rng(6).choice(nx * ny, cells, replace=False), repeat).astype(np.int64)
    prob.sources = sources(idx, (np.arange(idx.size) % 3).astype(np.int32), 4, 3)
    # six steps, sources for four: apart, two half steps, two source kernels
    # and the recording a step, then one launch (and the last recording);
    # inside, one launch
    assert same(fw2, prob, 6) == (4 * 5 + 2 if apart else 2)


@pytest.mark.parametrize("nx,ny,groups,apart", [
    (203, 77, [384, 1, 40], False), (203, 77, [3, 385], True), (203, 77, [203 * 77], True),
    (800, 700, [1] * (800 * 700), True), (800, 500, [1] * (800 * 500), False)])
def test_long_groups_and_dense_sensors_are_recorded_by_a_kernel_of_its_own(fw2, nx, ny, groups, apart):
    prob = problem(nx, ny, N=0, steps=5)
    k = sum(groups)
    idx = np.sort(np.random.default_rng(8).choice(nx * ny, k, replace=False)).astype(np.int64)
    prob.sensors = synth.Sensors(idx=idx, group=np.repeat(np.arange(len(groups)), groups).astype(np.int32),
                                 n_groups=len(groups))
    # seven steps with trace rows for five: apart, a launch and the recording
    # a step, then one launch; inside, one launch whose last step has no row
    assert same(fw2, prob, 7) == (5 * 2 + 1 if apart else 1)


class _GreenContext:
    """A stream that may use some of the device's SMs only (driver API)."""

    def __init__(self, sms):
        import ctypes as C
        import torch
        torch.cuda.current_stream().synchronize()          # the primary context exists
        self.C, self.cu = C, C.CDLL("libcuda.so.1")
        whole, part = (C.c_char * 144)(), (C.c_char * 144)()   # CUdevResource; the SM count at byte 96
        desc, self.ctx, self.ptr = C.c_void_p(), C.c_void_p(), C.c_void_p()
        dev, one = C.c_int(torch.cuda.current_device()), C.c_uint(1)
        self.call("cuDeviceGetDevResource", dev, whole, C.c_int(1))
        self.call("cuDevSmResourceSplitByCount", part, C.byref(one), whole, None, C.c_uint(0), C.c_uint(sms))
        self.sms = C.c_uint.from_buffer(part, 96).value
        self.call("cuDevResourceGenerateDesc", C.byref(desc), part, C.c_uint(1))
        self.call("cuGreenCtxCreate", C.byref(self.ctx), desc, dev, C.c_uint(1))
        self.call("cuGreenCtxStreamCreate", C.byref(self.ptr), self.ctx, C.c_uint(1), C.c_int(0))
        self.cuda_stream = self.ptr.value

    def call(self, name, *args):
        r = getattr(self.cu, name)(*args)
        if r == 801:
            pytest.skip("green contexts are not supported here")
        assert r == 0, f"{name}: {r}"

    def close(self):
        self.call("cuStreamSynchronize", self.ptr)
        self.call("cuStreamDestroy_v2", self.ptr)
        self.call("cuGreenCtxDestroy", self.ctx)


def test_stream_with_part_of_the_device_takes_half_steps_in_launches_of_their_own(fw2):
    """The blocks of a launch of many steps wait for one another; on a stream
    that holds some of the SMs they would not all be resident."""
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    prob = problem(600, 500)
    prob.sources = sources(np.arange(0, 600 * 500, 977, dtype=np.int64), np.zeros(308, np.int32), 4, 1)
    want, _ = run(fw2, prob, 6, "tile")
    green = _GreenContext(sms // 2)
    try:
        assert 0 < green.sms < sms
        sim = fw2.Simulation(prob, stream=green)
        sim.set_state(synth.random_state(prob, seed=4))
        before = sim.launches
        sim.step(6)
        assert sim.launches - before == 6 * 3               # two half steps and the recording a step
        sim.synchronize()
        for f, w in want.items():
            np.testing.assert_array_equal(sim.trace.cpu().numpy() if f == "trace" else sim.field(f), w, err_msg=f)
        sim.close()
    finally:
        green.close()


@pytest.mark.parametrize("maps", ["f32", "idx", "idx16"])
def test_half_steps_in_launches_of_their_own_with_sources_in_the_first_half_tiles(fw2, maps):
    """A launch copies its first half tiles while it looks up which of them
    hold sources and stages the index table: sources in every block's first
    and last half tile, one half step a launch, against the tile kernels."""
    prob = synth.indexed_abdominal_problem(nx=390, ny=1000, n_steps=12, n_elements=8, nl="literal", levels=64)
    if maps == "f32":
        prob = synth.abdominal_problem(n=256, n_steps=12, seed=3)
    elif maps == "idx16":
        prob.tissue = prob.tissue.astype(np.uint16)
    nx, ny = prob.shape
    cells = np.concatenate([np.arange(0, nx * ny, 1024), nx * ny - 1 - np.arange(40)]).astype(np.int64)
    prob.sources = [synth.Source(k, cells, np.zeros(cells.size, np.int32), a * np.ones((12, 1), np.float32))
                    for k, a in (("p", 10.0), ("vx", 1e-5), ("vy", 1e-5))]
    out = []
    for path in ("tile", "auto"):
        sim = fw2.Simulation(prob, map_precision=maps, kernel_path=path)
        for _ in range(12):
            fw2.fw2_step_part(sim.ctx, 0)
            fw2.fw2_step_part(sim.ctx, 1)
        sim.synchronize()
        assert fw2.fw2_kernel_path(sim.ctx) == ("tile" if path == "tile" else "pipe")
        out.append({f: sim.field(f) for f in ("p", "vx", "vy", "psi1x", "psi2y")})
        sim.close()
    assert np.abs(out[0]["p"]).max() > 0
    for f, w in out[0].items():
        np.testing.assert_array_equal(out[1][f], w, err_msg=f)


@pytest.mark.parametrize("N,nl,taps", [(3, "literal", False), (3, "pressure", True), (3, "literal", True), (2, "literal", True)])
def test_3d_batches_equal_their_contexts_alone_in_every_arithmetic_form(fw2, N, nl, taps):
    """The batched half steps of the register layout, two cells at a time or
    one, give the bits of the contexts stepped alone."""
    def sims():
        out = []
        for i, shape in enumerate(((140, 40, 24), (70, 33, 41))):
            prob = synth.homogeneous(shape, 1e-4, 0.0, relax=synth.relaxation_sets()[{2: "N2_y1.0_a0.5", 3: "N3_y1.2_brain"}[N]],
                                     beta=4.0)
            prob.c = (1500 + 100 * np.random.default_rng(i).random(prob.grid_shape)).astype(np.float32)
            prob.nl_mode, prob.dt = nl, 0.2 * 1e-4 / 2200.0
            prob.pml_transition, prob.pml_bound = 6, 2
            if taps:
                prob.taps = tuple(fw2.fw2_taps_time_space(0.25, 3))
            sim = fw2.Simulation(prob, map_precision="bf16")
            sim.set_state(synth.random_state(prob, seed=i))
            out.append(sim)
        return out
    alone, joined = sims(), sims()
    batch = fw2.fw2_batch_create([s.ctx for s in joined])
    fw2.fw2_batch_step(batch, 8)
    fw2.fw2_batch_synchronize(batch)
    for a, b in zip(alone, joined):
        a.step(8)
        a.synchronize()
        for f in ("p", "vx", "vz", "psi1x", "psi1z", "psi2y"):
            want = a.field(f)
            assert np.isfinite(want).all() and np.abs(want).max() > 0
            np.testing.assert_array_equal(b.field(f), want, err_msg=f)
    fw2.fw2_batch_destroy(batch)
    for s in alone + joined:
        s.close()


@pytest.mark.parametrize("maps", ["bf16", "f32"])
@pytest.mark.parametrize("shape", [(700, 240, 20), (500, 312, 20), (250, 640, 20)])   # six, four and two columns of units
def test_3d_rounds_over_the_blocks_reach_every_item(fw2, maps, shape):
    """More items than blocks, with the rounds rotated over the blocks (four
    and two columns) and not (six): the bits of the tile kernels."""
    from tests.test_gpu_parity import _pipe_vs_tile, small_3d
    prob = small_3d(n=shape, N=2, nl="pressure", steps=6, pml=(4, 1))
    _pipe_vs_tile(fw2, prob, 6, maps=maps, state=synth.random_state(prob, seed=2))
