"""Many time steps in one launch (2D pipelined path) against the same steps
taken half step by half step and against the tile kernels: the same bits.

The sizes cover one half tile, fewer half tiles than SMs, one round and a
ragged last round over the SMs, column counts that share factors with the SM
count, launches longer than the cap on steps per launch, several sources in
one cell and sensor groups across half tiles."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def fw2(fw2lib):
    from paper_2106_11476_gb300 import fw2 as m
    return m


def problem(nx, ny, N, nl, steps, seed=0):
    rng = np.random.default_rng(seed)
    sets = {0: None, 2: "N2_y1.0_a0.5", 3: "N3_y1.2_brain", 4: "N4_y1.1_a0.5"}[N]
    prob = synth.homogeneous((nx, ny), 1e-4, 0.0, relax=synth.relaxation_sets()[sets] if sets else None, beta=4.0)
    g = prob.grid_shape
    prob.c = (1500 + 100 * rng.random(g)).astype(np.float32)
    prob.rho = (1000 + 100 * rng.random(g)).astype(np.float32)
    prob.nl_mode = nl
    prob.dt = 0.3 * 1e-4 / 2200.0
    if N and min(nx, ny) >= 16:
        prob.pml_transition, prob.pml_bound = 5, 3
    # twelve cells of p (one of them twice) and, in v_x, v_y, a row and a column
    cells = rng.choice(nx * ny, size=min(12, nx * ny), replace=False).astype(np.int64)
    cells = np.concatenate([cells, cells[:1]])
    sig = rng.standard_normal((steps - 2, 3)).astype(np.float32)     # silent for the last two steps
    row, col = np.arange(nx, dtype=np.int64) + nx * (ny // 2), np.arange(ny, dtype=np.int64) * nx + nx // 3
    prob.sources = [synth.Source("p", cells, (np.arange(cells.size) % 3).astype(np.int32), 1e3 * sig),
                    synth.Source("vx", row, np.zeros(row.size, np.int32), 1e-3 * sig[:, :1]),
                    synth.Source("vy", col, np.zeros(col.size, np.int32), 1e-3 * sig[:, 1:2])]
    k = min(40, nx * ny)
    prob.sensors = synth.Sensors(idx=rng.choice(nx * ny, size=k, replace=False).astype(np.int64),
                                 group=np.sort(rng.integers(0, 5, k)).astype(np.int32), n_groups=5)
    prob.n_steps = steps - 1                                          # the last step has no trace row
    return prob


def run(fw2, prob, steps, how, path="auto"):
    sim = fw2.Simulation(prob, kernel_path=path)
    sim.set_state(synth.random_state(prob, seed=4))
    if how == "steps":
        sim.step(steps)
    else:
        for _ in range(steps):
            fw2.fw2_step_part(sim.ctx, 0)
            fw2.fw2_step_part(sim.ctx, 1)
    sim.synchronize()
    names = ["p", "vx", "vy"] + (["psi1x", "psi1y", "psi2x", "psi2y"] if prob.nrelax else [])
    out = {n: sim.field(n) for n in names}
    out["trace"] = sim.trace.cpu().numpy()
    sim.close()
    return out


@pytest.mark.parametrize("nx,ny,N,nl,steps", [
    (8, 8, 0, "off", 7), (120, 8, 2, "pressure", 7), (129, 9, 4, "literal", 7), (300, 200, 2, "westervelt", 9),
    (512, 304, 3, "off", 9), (1100, 515, 4, "pressure", 5), (2048, 160, 2, "off", 5), (64, 40, 2, "off", 519)])
def test_steps_in_one_launch_equal_half_steps_bitwise(fw2, nx, ny, N, nl, steps):
    prob = problem(nx, ny, N, nl, steps)
    ref = run(fw2, prob, steps, "steps", path="tile")
    assert np.abs(ref["p"]).max() > 0 and np.isfinite(ref["p"]).all()
    for how in ("steps", "parts"):
        got = run(fw2, prob, steps, how)
        for n, want in ref.items():
            np.testing.assert_array_equal(got[n], want, err_msg=f"{how}: {n}")


@pytest.mark.parametrize("maps", ["f16", "bf16"])
@pytest.mark.parametrize("nx,ny,N,nl,taps", [(129, 9, 0, "off", False), (203, 77, 2, "westervelt", True),
                                             (333, 140, 3, "off", False), (700, 260, 4, "literal", False)])
def test_16_bit_maps_on_the_pipelined_path_equal_tile_kernels_bitwise(fw2, maps, nx, ny, N, nl, taps):
    """FP16 (scaled) and bf16 maps staged by the pipelined kernels: odd widths,
    both sides of every C-PML strip, the cross taps and the literal system's K."""
    prob = problem(nx, ny, N, nl, 9, seed=2)
    if taps:
        prob.taps = tuple(fw2.fw2_taps_time_space(0.3))
    out = {}
    for path in ("tile", "auto"):
        sim = fw2.Simulation(prob, map_precision=maps, kernel_path=path)
        sim.set_state(synth.random_state(prob, seed=4))
        sim.step(9)
        assert fw2.fw2_kernel_path(sim.ctx) == ("tile" if path == "tile" else "pipe")
        out[path] = {n: sim.field(n) for n in ("p", "vx", "vy") + (("psi1x", "psi1y", "psi2x", "psi2y") if N else ())}
        out[path]["trace"] = sim.trace.cpu().numpy()
        sim.close()
    for n, want in out["tile"].items():
        np.testing.assert_array_equal(out["auto"][n], want, err_msg=n)


@pytest.mark.parametrize("levels,path", [(64, "pipe"), (369, "pipe"), (370, "tile")])
def test_uint16_index_takes_the_pipelined_path_while_its_tables_fit(fw2, levels, path):
    """1476 tissues of four mechanisms are the most that fit next to two
    stages; the same bits as the tile kernels on either side of the line."""
    prob = synth.indexed_abdominal_problem(nx=390, ny=220, n_steps=60, n_elements=8, nl="literal", levels=levels)
    prob.tissue = prob.tissue.astype(np.uint16)
    out = {}
    for p in ("tile", "auto"):
        sim = fw2.Simulation(prob, map_precision="idx16", kernel_path=p)
        sim.set_state(synth.random_state(prob, seed=4))
        sim.step(60)
        assert fw2.fw2_kernel_path(sim.ctx) == ("tile" if p == "tile" else path)
        out[p] = {n: sim.field(n) for n in ("p", "vx", "vy", "psi1x", "psi2y")}
        sim.close()
    for n, want in out["tile"].items():
        np.testing.assert_array_equal(out["auto"][n], want, err_msg=n)


@pytest.mark.parametrize("n,N,nl,pml,taps", [
    ((300, 70, 45), 3, "westervelt", (6, 2), False), ((300, 70, 45), 3, "literal", (6, 2), True),
    ((300, 60, 20), 0, "off", (0, 0), True), ((200, 45, 30), 2, "pressure", (5, 2), True),
    ((100, 40, 20), 2, "literal", (6, 2), False), ((200, 20, 17), 3, "off", (3, 1), False),
    ((300, 600, 20), 1, "off", (6, 2), False)])
def test_3d_float_maps_on_the_pipelined_path_equal_tile_kernels_bitwise(fw2, n, N, nl, pml, taps):
    """Float maps staged by the 3D pipeline: interior and edge units, one x
    tile reaching both strips, strips read per cell (5 + 2 cells), few planes,
    more items than blocks, the cross taps and the literal system's K."""
    from tests.test_gpu_parity import _pipe_vs_tile, small_3d
    prob = small_3d(n=n, N=max(N, 1), nl=nl, steps=12, pml=pml)
    if N == 0:
        prob.nrelax = 0
        prob.kappa1 = prob.kappa2 = prob.d1 = prob.alpha1 = prob.d2 = prob.alpha2 = None
    prob.sensors = synth.random_sensors(n, 25, 4, np.random.default_rng(1))
    prob.sources = [synth.Source("p", np.arange(60, dtype=np.int64) * 11, np.zeros(60, np.int32),
                                 prob.sources[0].signal)]
    if taps:
        prob.taps = tuple(fw2.fw2_taps_time_space(0.35, 3))
    _pipe_vs_tile(fw2, prob, 12, maps="f32", state=synth.random_state(prob, seed=21))


@pytest.mark.parametrize("shape,offset", [((8, 8), 0), ((33, 9), 0), ((1024, 8), 0), ((1028, 11), 1), ((2051, 16), 0),
                                          ((17, 9, 8), 0), ((64, 8, 10), 3)])
def test_device_field_copies_round_trip(fw2, shape, offset):
    """Fields to and from device buffers of any row alignment (rows of 4n and
    odd lengths, longer than a segment, buffers off by `offset` floats) equal
    the copies through host memory; what lies beside the buffer is untouched."""
    import torch
    prob = synth.homogeneous(shape, 1e-4, 2e-8, relax=synth.relaxation_sets()["N2_y1.0_a0.5"])
    sim = fw2.Simulation(prob)
    rng = np.random.default_rng(7)
    for name in ("p", "v" + "xyz"[len(shape) - 1], "psi1x", "psi2y"):
        g = ((2,) if name.startswith("psi") else ()) + prob.grid_shape
        n = int(np.prod(g))
        want = rng.standard_normal(n).astype(np.float32)
        buf = torch.full((n + offset + 8,), -7.0, device="cuda")
        buf[offset:offset + n] = torch.from_numpy(want).cuda()
        fw2.fw2_set_field(sim.ctx, name, buf[offset:offset + n])
        np.testing.assert_array_equal(sim.field(name).ravel(), want)
        got = torch.full((n + offset + 8,), -7.0, device="cuda")
        fw2.fw2_get_field(sim.ctx, name, got[offset:offset + n])
        assert torch.equal(got, buf)
        if not name.startswith("psi"):
            rows = prob.grid_shape[0]
            part = torch.empty((rows - 3,) + prob.grid_shape[1:], device="cuda")
            fw2.fw2_get_rows(sim.ctx, name, 2, rows - 3, part)
            np.testing.assert_array_equal(part.cpu().numpy(), want.reshape(g)[2:rows - 1])
    sim.close()
