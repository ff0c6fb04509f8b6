"""Performance cases of the Fullwave 2 stepper: what its users have it do.

A pass is what a simulation loop does between two looks at its data: advance
a context (or a batch of contexts, or a request from its medium to its
traces) a number of time steps through the public calls, sources firing and
sensors recording, and copy the fields out.  The grids, media, source arrays,
mechanism counts, C-PML thicknesses and storage forms follow the repository's
configurations: 2D soft tissue at 12 points per wavelength of 3 MHz with a
3 + 1 wavelength C-PML, 3D transcranial media at 10 points per wavelength of
1 MHz with 40 boundary cells.  Contexts start from a smooth seeded wavefield,
so every cell does work from the first step.

`exact` advances the same inputs with plain torch operations in 64 bits:
coefficients from the closed forms, the storage rounding that the caller
chose (bf16 and FP16 maps), no fusion and no tiling.
"""
from __future__ import annotations

import math
from types import SimpleNamespace

import torch

from paper_2106_11476_gb300 import fw2

# Fitted relaxation sets (power law alpha0 f^y, N mechanisms) of the
# repository's workloads: kappa1, kappa2, d1, alpha1, d2, alpha2 [1/s].
SETS = {
    "soft2": (0.901183277, 1.10165141, [28015.2191, 4760.13255], [9547270.42, 100000.0],
              [131719.846, 1226677.11], [45453026.8, 256477804.0]),
    "brain3": (0.812774423, 1.18302663, [20937.3099, 100.0, 31130988.7], [7405196.89, 1.0e12, 2205842690.0],
               [766002.0, 129311.324, 11917287.7], [115248522.0, 30189063.5, 928073662.0]),
    "skull3": (0.804561287, 0.855526566, [321138.988, 2146590.45, 63072341.3], [10636114.8, 58058994.3, 285345032.0],
               [153014.399, 836902.161, 21960.2284], [1413388.46, 29283121.1, 495656728.0]),
    "fat4": (0.839227514, 1.17359187, [46963.2114, 8156632.64, 12387.115, 258911.999],
             [23129856.0, 989042450.0, 5099804.46, 114845401.0], [286.449006, 70308.3695, 2139620.62, 100.0],
             [100000.0, 62511102.3, 7219850630.0, 1.0e12]),
    "muscle4": (0.894115227, 1.09292807, [3559129.4, 1243.77176, 100.0, 23731.5448],
                [305585549.0, 1.0e12, 1.0e12, 2774025.23], [98236.6269, 403296.536, 668877.226, 3074445.3],
                [15842926.3, 57635437.3, 359461352.0, 21448007600.0]),
    "connective4": (0.816753242, 1.18442693, [100.0, 4918653.91, 291223.386, 412.019825],
                    [1.0e12, 276194778.0, 41414576.1, 100000.0], [206715.43, 100.0, 119728.435, 19875.4655],
                    [72196514.2, 1.0e12, 9493917.04, 100000.0]),
}
# c [m/s], rho [kg/m^3], beta, relaxation set, scale of d^(nu=1)
SOFT4 = [(1540.0, 1000.0, 3.5, "fat4", 0.042), (1478.0, 950.0, 6.0, "fat4", 1.0),
         (1547.0, 1050.0, 4.6, "muscle4", 1.0), (1613.0, 1120.0, 5.0, "connective4", 1.0)]
SOFT2 = [(1540.0, 1000.0, 3.5, "soft2", 0.04), (1478.0, 950.0, 6.0, "soft2", 0.96),
         (1547.0, 1050.0, 4.6, "soft2", 2.18), (1613.0, 1120.0, 5.0, "soft2", 3.14)]
HEAD3 = [(1560.0, 1040.0, 4.5, "brain3", 1.0), (2550.0, 1775.0, 4.5, "skull3", 0.9),
         (2700.0, 1850.0, 4.5, "skull3", 1.0), (2900.0, 1950.0, 4.5, "skull3", 1.2)]
CLASSES = {2: SOFT2, 3: HEAD3, 4: SOFT4}

FIELDS = {2: ("p", "vx", "vy"), 3: ("p", "vx", "vy", "vz")}
MEMORY = {2: ("psi1x", "psi1y", "psi2x", "psi2y"),
          3: ("psi1x", "psi1y", "psi1z", "psi2x", "psi2y", "psi2z")}
# contexts of up to this many cells also return their memory variables (a
# whole checkpoint of the state)
CHECKPOINT_CELLS = 1 << 22
TAYLOR = (1225.0 / 1024.0, -245.0 / 3072.0, 49.0 / 5120.0, -5.0 / 7168.0, 0.0)


def _case(name, what, shape, n_relax, maps, nl, steps, taps="taylor", n_ctx=1):
    c = {"what": what, "nx": shape[0], "ny": shape[1], "nz": shape[2] if len(shape) > 2 else 1, "n_relax": n_relax,
         "maps": maps, "nl": nl, "taps": taps, "steps": steps, "n_ctx": n_ctx}
    return {"name": name, **c} if name else c


def listed():
    return [
        # a first look at a setup: a small linear grid, where launches and
        # latency are everything
        _case("quick-2d", "run", (250, 186), 2, "f32", "off", 200),
        # the plain 2D method: 512^2, four mechanisms, linear
        _case("plain-2d", "run", (512, 512), 4, "f32", "off", 200),
        # an imaging crop of odd size with the time-space optimised taps
        _case("ragged-2d", "run", (1501, 1237), 4, "f32", "westervelt", 24, taps="ts"),
        # the whole abdominal wall, nonlinear: the largest 2D grid
        _case("abdominal-2d", "run", (4096, 4096), 4, "f32", "pressure", 4),
        # one transmit over a medium stored as a uint8 tissue index
        _case("index-2d", "run", (2048, 1024), 4, "idx", "pressure", 24),
        # a medium of more than 256 tissues: uint16 index
        _case("index16-2d", "run", (1536, 2048), 4, "idx16", "pressure", 16),
        # FP16 maps, the reduced storage of a medium without tissue classes
        _case("half-2d", "run", (1800, 1100), 4, "f16", "pressure", 16),
        # the transmits of a sequence in one batch, uneven sizes
        _case("batch-2d", "batch", (2048, 1024), 4, "idx", "pressure", 32, n_ctx=6),
        # a whole request: new medium in, coefficient build, steps, traces out
        _case("request-2d", "request", (1024, 768), 4, "f32", "pressure", 40),
        # a served 3D request with bf16 maps, sizes that fit no tile
        _case("ragged-3d", "run", (301, 222, 190), 3, "bf16", "pressure", 8),
        # the plain 3D form: float maps, the default storage
        _case("plain-3d", "run", (256, 256, 256), 3, "f32", "off", 5),
        # the transcranial medium with bf16 maps: the largest case
        _case("skull-3d", "run", (512, 512, 512), 3, "bf16", "off", 4),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _steps(cells, full, most):
    return max(4, min(most, int(full / cells)))


def draw(rng):
    kind = rng.choice(["plain", "plain", "index", "stored", "batch", "request", "head", "head32"])
    nl = rng.choice(["off", "pressure", "pressure", "westervelt", "literal"])
    taps = rng.choice(["taylor", "taylor", "ts"])
    if kind in ("plain", "index", "stored"):
        nx, ny = _log(rng, 100, 4096), _log(rng, 100, 4096)
        if kind == "plain":
            maps, n_relax = "f32", rng.choice([2, 3, 4, 4])
        elif kind == "index":
            maps, n_relax = "idx", rng.choice([2, 3, 4, 4])
        else:
            maps, n_relax = rng.choice(["idx16", "f16", "bf16"]), rng.choice([2, 3, 4, 4])
        return _case(None, "run", (nx, ny), n_relax, maps, nl, _steps(nx * ny, 6.4e7, 200), taps)
    if kind == "batch":
        nx, ny, n_ctx = _log(rng, 512, 2048), _log(rng, 512, 1024), rng.randint(2, 8)
        return _case(None, "batch", (nx, ny), 4, rng.choice(["idx", "idx", "f32"]), nl,
                     _steps(nx * ny * n_ctx, 4e8, 48), taps, n_ctx)
    if kind == "request":
        nx, ny = _log(rng, 256, 2048), _log(rng, 256, 2048)
        return _case(None, "request", (nx, ny), rng.choice([2, 4]), rng.choice(["f32", "f32", "idx"]), nl,
                     _steps(nx * ny, 3.2e7, 100), taps)
    hi, full = (400, 9e7) if kind == "head" else (200, 3e7)
    shape = [_log(rng, 100, hi) for _ in range(3)]
    return _case(None, "run", shape, 3, "bf16" if kind == "head" else "f32", nl,
                 _steps(shape[0] * shape[1] * shape[2], full, 40), taps)


def _shape(case):
    return (case["nx"], case["ny"]) if case["nz"] == 1 else (case["nx"], case["ny"], case["nz"])


def _members(case):
    """Grid of each context of the case: a batch holds whole crops and, every
    third context, a smaller instance."""
    nx, ny = case["nx"], case["ny"]
    if case["what"] != "batch":
        return [_shape(case)]
    return [(nx, ny) if i % 3 < 2 else (max(256, nx * 5 // 9 + 7 * i), max(256, ny * 3 // 4 - 5 * i))
            for i in range(case["n_ctx"])]


# ------------------------------------------------------------------ inputs ---

def _wave(shape, gen, scale, dev):
    """A smooth wavefield: three plane waves of at least eight cells per
    wavelength, float32 [..., y, x]."""
    out = torch.zeros(tuple(reversed(shape)), device=dev)
    nd = len(shape)
    for _ in range(3):
        u = torch.rand(nd + 2, generator=gen, device="cpu").tolist()
        arg = torch.full((1,) * nd, 2 * math.pi * u[nd], device=dev)
        for q in range(nd):
            view = [1] * nd
            view[nd - 1 - q] = shape[q]
            arg = arg + ((2 * u[q] - 1) * 2 * math.pi / 8) * torch.arange(shape[q], device=dev).view(view)
        out += (scale * (0.3 + u[nd + 1])) * torch.sin(arg)
    return out


def _class_map(shape, gen, dev):
    """Tissue class 0 .. 3 of every cell: wavy layers under a coupling layer in
    2D, an ellipsoidal shell with smooth porosity in 3D."""
    if len(shape) == 2:
        nx, ny = shape
        x = torch.arange(nx, device=dev, dtype=torch.float32)
        y = torch.arange(ny, device=dev, dtype=torch.float32).view(ny, 1)
        cls = torch.zeros((ny, nx), dtype=torch.int64, device=dev)
        depth = 56.0
        while depth < ny:
            u = torch.rand(4, generator=gen, device="cpu").tolist()
            surface = depth + 6.0 * torch.sin(0.03 * (1 + u[0]) * x + 6.3 * u[1]) + 3.0 * torch.sin(0.11 * x + 6.3 * u[2])
            cls = torch.where(y >= surface, torch.full_like(cls, 1 + int(3 * u[3])), cls)
            depth += 47 + 70 * u[0]
        return cls
    nx, ny, nz = shape
    c = [(torch.arange(s, device=dev, dtype=torch.float32) - (s - 1) / 2) / (a * s)
         for s, a in zip(shape, (0.40, 0.36, 0.32))]
    r = torch.sqrt(c[0].view(1, 1, nx) ** 2 + c[1].view(1, ny, 1) ** 2 + c[2].view(nz, 1, 1) ** 2)
    shell = (r >= 1.0) & (r < 1.06)
    poro = _wave(shape, gen, 1.0, dev)
    level = 1 + (poro > -0.4).to(torch.int64) + (poro > 0.5).to(torch.int64)
    return torch.where(shell, level, torch.zeros_like(level))


def _problem(case, shape, seed):
    """One problem, its arrays on the GPU (the attributes fw2.Simulation takes)
    and its starting fields."""
    dev = "cuda"
    gen = torch.Generator(device="cpu")
    gen.manual_seed(int(seed) * 7919 + 17)
    gpu = torch.Generator(device=dev)
    gpu.manual_seed(int(seed) * 104729 + 5)
    nd, N = len(shape), case["n_relax"]
    f0, ppw, c0 = (3e6, 12.0, 1540.0) if nd == 2 else (1e6, 10.0, 1540.0)
    h = c0 / f0 / ppw
    lt, lb = (36, 12) if nd == 2 else (30, 10)
    table = CLASSES[N]
    cls = _class_map(shape, gen, dev)
    indexed = case["maps"] in ("idx", "idx16")
    # scatterers: 20 per squared wavelength in 2D, +-2 % on c and rho, clipped
    # at 8 %; the index forms quantise them to a number of levels per class
    levels = {"idx": 64, "idx16": 290}.get(case["maps"], 0)
    pert = torch.randn(cls.shape, generator=gpu, device=dev).mul_(0.02).clamp_(-0.0799, 0.0799)
    pert *= (torch.rand(cls.shape, generator=gpu, device=dev) < 20.0 / (ppw * ppw)) & (cls > 0)
    rows = {"c": [], "rho": [], "beta": [], "kappa1": [], "kappa2": [], "d1": [], "alpha1": [], "d2": [], "alpha2": []}
    for c, rho, beta, key, scale in table:
        k1, k2, d1, al1, d2, al2 = SETS[key]
        for lv in range(max(levels, 1)):
            f = 1.0 if lv == 0 else 0.92 + 0.16 * (lv - 1) / (levels - 2)
            for k, v in (("c", c * f), ("rho", rho * f), ("beta", beta), ("kappa1", k1), ("kappa2", k2),
                         ("d1", [d1[0] * scale] + d1[1:]), ("alpha1", al1), ("d2", [d2[0] * scale] + d2[1:]),
                         ("alpha2", al2)):
                rows[k].append(v)
    tab = {k: torch.tensor(v, dtype=torch.float32, device=dev) for k, v in rows.items()}
    for k in ("d1", "alpha1", "d2", "alpha2"):
        tab[k] = tab[k].t().contiguous()
    pr = SimpleNamespace(shape=shape, h=h, nrelax=N, pml_transition=lt, pml_bound=lb, pml_rc=1e-3, pml_npow=2.0,
                         pml_reading="C", nl_mode=case["nl"], memory_alignment="centred", bc=("zero",) * 3,
                         taps=None, tissue=None, tables=None)
    if indexed:
        lv = torch.where(pert != 0, ((pert + 0.08) / 0.16 * (levels - 2)).round().to(torch.int64) + 1,
                         torch.zeros_like(cls)).clamp_(0, levels - 1)
        idx = cls * levels + lv
        pr.tissue = idx.to(torch.uint8) if case["maps"] == "idx" else idx.to(torch.int16)
        pr.tables = tab
        cells = (tab["c"][idx], tab["rho"][idx])
        del idx, lv
        smax = float((tab["c"] / torch.sqrt(tab["kappa1"] * tab["kappa2"])).double().max())
        pr.pml_cp = float(cells[0].max())
    else:
        pr.c = tab["c"][cls] * (1 + pert)
        pr.rho = tab["rho"][cls] * (1 + pert)
        pr.beta = tab["beta"][cls] if case["nl"] != "off" else None
        for k in ("kappa1", "kappa2"):
            setattr(pr, k, tab[k][cls])
        for k in ("d1", "alpha1", "d2", "alpha2"):
            setattr(pr, k, torch.stack([tab[k][n][cls] for n in range(N)]))
        smax = float((pr.c / torch.sqrt(pr.kappa1 * pr.kappa2)).double().max())
        pr.pml_cp = float(pr.c.max())
    del pert, cls
    pr.dt = 0.4 * h / smax
    if case["taps"] == "ts":
        pr.taps = fw2.fw2_taps_time_space(0.4 * c0 / smax, nd)
    # a linear (3D: planar) array of up to 64 (3D: 16 x 16) elements, each a
    # source column with its own delay and a sensor group
    L = lt + lb
    steps = case["steps"]
    if nd == 2:
        n_el = max(1, min(64, (shape[0] - 2 * L) // 12))
        x0 = max(L, (shape[0] - 12 * n_el) // 2)
        e, w = torch.meshgrid(torch.arange(n_el), torch.arange(11), indexing="ij")
        xs = (x0 + 12 * e + w).reshape(-1).clamp_(max=shape[0] - 1)
        cell = xs + shape[0] * min(L + 4, shape[1] - 1)
        group = e.reshape(-1)
        off = (torch.arange(n_el) - (n_el - 1) / 2) * 12 * h
        delay = (math.hypot(float(off.abs().max()), 0.03) - torch.sqrt(off.double() ** 2 + 0.03 ** 2)) / c0
        amp = 1.0e5
    else:
        n_el, pitch = 256, 5
        a = torch.arange(16 * pitch)
        a = a[a % pitch < pitch - 1]
        y, x = torch.meshgrid(a, a, indexing="ij")
        cell = ((shape[0] // 2 - 40 + x).clamp(0, shape[0] - 1) + shape[0] * ((shape[1] // 2 - 40 + y).clamp(0, shape[1] - 1)
                + shape[1] * min(L + 4, shape[2] - 1))).reshape(-1)
        group = (16 * (y // pitch) + x // pitch).reshape(-1)
        delay = torch.zeros(n_el, dtype=torch.float64)
        amp = 1.0e4
    t = (torch.arange(steps, dtype=torch.float64) + 1).view(-1, 1) * pr.dt - delay.view(1, -1) - 0.3 / f0
    sig = amp * torch.exp(-(t * f0 / 1.5) ** 2) * torch.sin(2 * math.pi * f0 * t)
    pr.sources = [SimpleNamespace(kind="p", idx=cell.to(torch.int64).numpy(), group=group.to(torch.int32).numpy(),
                                  signal=sig.to(torch.float32).numpy())]
    pr.sensors = SimpleNamespace(idx=pr.sources[0].idx, group=pr.sources[0].group, n_groups=n_el)
    pr.n_steps = steps
    pr.start = {"p": _wave(shape, gen, 1e5, dev)}
    for q in range(nd):
        pr.start["v" + "xyz"[q]] = _wave(shape, gen, 1e5 / (1000.0 * 1540.0), dev)
    return pr


def _outputs(case, shape):
    nd, N = len(shape), case["n_relax"]
    g = tuple(reversed(shape))
    out = {f: torch.empty(g, device="cuda") for f in FIELDS[nd]}
    if math.prod(shape) <= CHECKPOINT_CELLS:
        out.update({f: torch.empty((N,) + g, device="cuda") for f in MEMORY[nd]})
    return out


def _simulation(case, pr, start=True):
    sim = fw2.Simulation(pr, map_precision=case["maps"])
    if start:
        sim.set_state(pr.start)
    return sim


class _State:
    """Contexts, the batch over them and the buffers their fields come out into."""

    def __init__(self, case, problems):
        self.case = case
        self.batch = None
        self.sims = []
        if case["what"] == "request":
            self.problem = problems[0]
            self.out = [_outputs(case, problems[0].shape)]
            return
        shapes = [p.shape for p in problems]
        while problems:
            pr = problems.pop(0)
            self.sims.append(_simulation(case, pr))
            # the context holds its own maps and state from here on
            for k in ("c", "rho", "beta", "kappa1", "kappa2", "d1", "alpha1", "d2", "alpha2", "tissue", "start"):
                setattr(pr, k, None)
        self.out = [_outputs(case, s) for s in shapes]
        if case["what"] == "batch":
            self.batch = fw2.fw2_batch_create([s.ctx for s in self.sims])

    def __del__(self):
        try:
            if self.batch:
                fw2.fw2_batch_destroy(self.batch)
                self.batch = None
            for s in self.sims:
                s.close()
        except Exception:
            pass


def prepare(case, seed):
    return _State(case, [_problem(case, s, seed + 1009 * i) for i, s in enumerate(_members(case))])


def _read(sim, out):
    for name, buf in out.items():
        fw2.fw2_get_field(sim.ctx, name, buf)
    return {"trace": sim.trace, **out}


def run(state):
    case = state.case
    n = case["steps"]
    if case["what"] == "request":
        sim = _simulation(case, state.problem)
        sim.step(n)
        got = _read(sim, state.out[0])
        sim.close()
        return got
    for sim in state.sims:
        fw2.fw2_set_step(sim.ctx, 0)      # the transmit fires and the traces start at row 0
    if state.batch:
        fw2.fw2_batch_step(state.batch, n)
        fw2.fw2_batch_synchronize(state.batch)
    else:
        state.sims[0].step(n)
    got = [_read(sim, out) for sim, out in zip(state.sims, state.out)]
    return got if state.batch else got[0]


def work(case):
    """Of every time step: the state read and written once, every map and
    C-PML strip read once (the index forms: the index, per half step), the
    fields read once per output."""
    nd, N = (2, case["n_relax"]) if case["nz"] == 1 else (3, case["n_relax"])
    e = {"f32": 4, "bf16": 2, "f16": 2}.get(case["maps"], 0)
    i = {"idx": 1, "idx16": 2}.get(case["maps"], 0)
    L, es = (48 if nd == 2 else 40), e or 4
    nl = 1 if case["nl"] != "off" else 0
    total_b = total_f = 0.0
    for shape in _members(case):
        cells = math.prod(shape)
        step = cells * (8 * (1 + nd + 2 * nd * N) + 2 * i + e * (4 + nl + 4 * N))
        step += sum(min(2 * L, s) * (cells // s) for s in shape) * 4 * N * es
        outs = 1 + nd + (2 * nd * N if cells <= CHECKPOINT_CELLS else 0)
        total_b += case["steps"] * step + 8.0 * cells * outs
        if case["what"] == "request":
            total_b += 4.0 * cells * (4 + nl + 4 * N) if e else cells * i
        taps = 12 + (8 * (nd - 1) if case["taps"] == "ts" else 0)
        total_f += case["steps"] * cells * (2 * nd * (taps + 1 + 7 * N) + 5 * nd + 6 + 3 * nl)
    return {"bytes": total_b, "flops": total_f}


# ------------------------------------------------------------------- exact ---

def _stored(maps, *values):
    """The values as the chosen storage holds them (FP16: each divided by one
    power of two that puts the largest of all in [2^14, 2^15))."""
    if maps == "bf16":
        return [v.to(torch.float32).to(torch.bfloat16).double() for v in values]
    if maps == "f16":
        m = max(float(v.abs().max().to(torch.float32)) for v in values)
        s = math.ldexp(1.0, math.frexp(m)[1] - 15) if m > 0 else 1.0
        return [(v / s).to(torch.float32).to(torch.float16).double() * s for v in values]
    return list(values)


def _profile(X0, depth, nu, is_d, lt, lb, d_target):
    """A relaxation parameter inside the two-stage C-PML at `depth` cells (0 in
    the interior), X0 the tissue's value."""
    L = lt + lb
    g_t = torch.where(depth < lt, 0.5 * (1 - torch.cos(math.pi * depth / lt)), torch.ones_like(depth))
    if nu == 0 and is_d:
        v = (d_target - X0) * (depth / L) ** 2 + X0
    elif nu == 0:
        v = (1 - g_t) * X0 + g_t * (d_target * (1 - depth / L))
    else:
        v = X0 - X0 * g_t
    return torch.where(depth > 0, v, X0)


def _ab(d, al, kappa, dt):
    em = torch.expm1(-(d / kappa + al) * dt)
    den = kappa * (d + kappa * al)
    return torch.where((d == 0) | (den == 0), torch.zeros_like(em), d * em / den), em


def _shift(f, ax, s):
    """g[i] = f[i + s] along ax, zero outside."""
    out = torch.zeros_like(f)
    n = f.shape[ax]
    if abs(s) < n:
        out.narrow(ax, max(0, -s), n - abs(s)).copy_(f.narrow(ax, max(0, s), n - abs(s)))
    return out


def _diff(f, ax, taps, h, face):
    """Staggered derivative along axis ax at the +1/2 faces or, of a face
    field, at the centres."""
    D = torch.zeros_like(f)
    for m in range(1, 5):
        hi, lo = (m, 1 - m) if face else (m - 1, -m)
        D += (taps[m - 1] / h) * (_shift(f, ax, hi) - _shift(f, ax, lo))
    if taps[4] != 0:
        g = _shift(f, ax, 1) - f if face else f - _shift(f, ax, -1)
        for t in range(f.dim()):
            if t != ax:
                D += (taps[4] / h) * (_shift(g, t, 1) + _shift(g, t, -1))
    return D


def _advance(case, pr):
    nd, N, dt, h, maps = len(pr.shape), pr.nrelax, pr.dt, pr.h, case["maps"]
    if pr.tissue is not None:
        at = pr.tissue.to(torch.int64)
        cell = lambda k, n=None: (pr.tables[k] if n is None else pr.tables[k][n])[at].double()
    else:
        cell = lambda k, n=None: (getattr(pr, k) if n is None else getattr(pr, k)[n]).double()
    c, rho = cell("c"), cell("rho")
    K = rho * c * c
    chi = None
    if pr.nl_mode != "off":
        chi = (-2.0 * cell("beta") if pr.nl_mode == "westervelt" else 1.0 - 2.0 * cell("beta")) / K
        chi, = _stored(maps, chi)
    K, = _stored(maps, K)
    rho, = _stored(maps, rho)
    del c
    k1, k2 = cell("kappa1"), cell("kappa2")
    ik1, = _stored(maps, 1.0 / k1)
    ik2, = _stored(maps, 1.0 / k2)
    lt, lb = pr.pml_transition, pr.pml_bound
    L = lt + lb
    d_target = -3.0 * pr.pml_cp * math.log(pr.pml_rc) / (2.0 * L * h)

    def next_cell(f, ax):        # the +1 neighbour; the last cell its own
        n = f.shape[ax]
        return torch.cat([f.narrow(ax, 1, n - 1), f.narrow(ax, n - 1, 1)], ax)

    def coefficients(op):        # [axis][nu] -> (a, b - 1)
        kap, dn, an = (k1, "d1", "alpha1") if op == 1 else (k2, "d2", "alpha2")
        out = [[None] * N for _ in range(nd)]
        for nu in range(N):
            d, al = cell(dn, nu), cell(an, nu)
            ab = [_ab(d, al, kap, dt)] if maps == "f16" else []   # the tissue's own take part in the scale
            for q in range(nd):
                n = pr.shape[q]
                x = torch.arange(n, dtype=torch.float64, device=d.device) + (0.5 if op == 1 else 0.0)
                depth = torch.clamp(torch.maximum(L - 0.5 - x, x - (n - L - 0.5)), 0.0, float(L))
                view = [1] * nd
                view[nd - 1 - q] = n
                depth = depth.view(view)
                ab.append(_ab(_profile(d, depth, nu, True, lt, lb, d_target),
                              _profile(al, depth, nu, False, lt, lb, d_target), kap, dt))
            a, b = _stored(maps, *[v[0] for v in ab]), _stored(maps, *[v[1] for v in ab])
            for q in range(nd):
                out[q][nu] = (a[q - nd], b[q - nd])
        return out

    ab1, ab2 = coefficients(1), coefficients(2)
    del k1, k2
    p = pr.start["p"].double()
    v = [pr.start["v" + "xyz"[q]].double() for q in range(nd)]
    psi = {op: [[torch.zeros_like(p) for _ in range(N)] for _ in range(nd)] for op in (1, 2)}

    def stretched(D, op, q, ik):
        S = D * ik
        for nu in range(N):
            a, b = (ab1 if op == 1 else ab2)[q][nu]
            old = psi[op][q][nu]
            new = old + b * old + a * D
            S += 0.5 * (new + old)
            psi[op][q][nu] = new
        return S

    taps = pr.taps if pr.taps is not None else TAYLOR
    src, sen = pr.sources[0], pr.sensors
    at_src, grp = torch.from_numpy(src.idx).to(p.device), torch.from_numpy(src.group).to(p.device).long()
    signal = torch.from_numpy(src.signal).to(p.device).double()
    count = torch.zeros(sen.n_groups, dtype=torch.float64, device=p.device).index_add_(
        0, grp, torch.ones_like(grp, dtype=torch.float64))
    trace = torch.zeros((pr.n_steps, sen.n_groups), dtype=torch.float64, device=p.device)
    for n in range(pr.n_steps):
        for q in range(nd):
            ax = nd - 1 - q
            S = stretched(_diff(p, ax, taps, h, True), 1, q, ik1)
            if pr.nl_mode == "literal":
                S = S / (1.0 + 0.5 * (1.0 / K + 1.0 / next_cell(K, ax)) * 0.5 * (p + _shift(p, ax, 1)))
            v[q] = v[q] - (2.0 * dt / (rho + next_cell(rho, ax))) * S
        div = sum(stretched(_diff(v[q], nd - 1 - q, taps, h, False), 2, q, ik2) for q in range(nd))
        upd = dt * K * div
        p = p - (upd if chi is None else upd / (1.0 + chi * p))
        p.view(-1).index_add_(0, at_src, signal[n][grp])
        trace[n] = torch.zeros_like(count).index_add_(0, grp, p.reshape(-1)[at_src]) / torch.clamp(count, min=1.0)
    out = {"trace": trace, "p": p, **{"v" + "xyz"[q]: v[q] for q in range(nd)}}
    if math.prod(pr.shape) <= CHECKPOINT_CELLS:
        for q in range(nd):
            out["psi1" + "xyz"[q]] = torch.stack(psi[1][q])
            out["psi2" + "xyz"[q]] = torch.stack(psi[2][q])
    return out


def exact(case, seed):
    got = [_advance(case, _problem(case, s, seed + 1009 * i)) for i, s in enumerate(_members(case))]
    return got if case["what"] == "batch" else got[0]
