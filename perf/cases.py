"""The work that users of the RRMHD lattice Boltzmann library have it do, as
measurable cases: time stepping of 1-D, 2-D and 3-D runs through `Solver` (one
run, a few equal runs, a sweep of uneven runs; every storage precision; periodic,
open and driven faces; plain, Gauss-charge and learned-seed recovery) with the
read-out of the fields a program does between its steps, and the training,
gradient and inference of the learned recovery seed.

`exact` restates the method (arXiv:1508.03452, Sec. III) in plain float64
tensors, independent of the library.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1508_03452_gb300 import lbrmhd as L

PRECISION = {"fp64": L.FP64, "fp32": L.FP32, "fp16": L.FP16_DEV}
# snapshots are kept in the type of the run's storage
SNAPSHOT = {"fp64": torch.float64, "fp32": torch.float32, "fp16": torch.float16}
BYTES_PER_UPDATE = {"fp64": 1200, "fp32": 600, "fp16": 448}  # 63 populations + 12 primitives, in and out once
FLOPS_PER_UPDATE = {1: 1500, 2: 1900, 3: 2400}  # streaming, moments, recovery (two passes), collision
GAMMA_AD, TAU = 4.0 / 3.0, 1.0


def sim(kind, name=None, **kw):
    """A stepping case: `runs` runs of one kind in a handle, `steps` steps and a
    snapshot of every run a pass. `fresh`: a pass is a whole experiment, from the
    initial fields on ("host": numpy arrays, "device": tensors); otherwise ("") it is
    the next interval of a longer run."""
    c = dict(kind=kind, nx=1, ny=1, nz=1, runs=1, precision="fp32", steps=10, sigma=100.0, alpha=0.1, c=1.0, dx=1.0,
             gauss=False, learned=False, fresh="", monitor=False, streams=1, graph=0)
    c.update(kw)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the paper's own 1-D current-sheet test from t = 1 to t = 9, whole: the smallest run there is, in the
        # precision its convergence study needs; two dependent launches a step
        sim("sheet1d", "sheet_1d_100_fp64", nx=100, precision="fp64", steps=377, dx=0.03, fresh="host"),
        # a linear Alfven wave on the small box of the correctness runs, stepped as it comes (default schedule)
        sim("alfven", "alfven_64_fp32", nx=64, ny=64, steps=100, sigma=1e4),
        # the benchmark's workload: three conductivities of the 1024^2 current sheet in one handle, the schedule
        # the autotuner picks for it
        sim("sheet", "sheets_3x1024_fp32", nx=1024, ny=1024, runs=3, steps=20, streams=3, graph=10),
        # large shear layers in the float16-deviation storage (fewest bytes)
        sim("kh", "kh_2048_fp16", nx=2048, ny=2048, precision="fp16", steps=10, alpha=0.02, gauss=True),
        # a float64 reference run of a ragged box
        sim("sheet", "sheet_509x387_fp64", nx=509, ny=387, precision="fp64", steps=5),
        # the flare set-up from its initial fields on: the largest grid, open faces, driven bottom
        sim("rope", "rope_256_fp32", nx=256, ny=256, nz=256, steps=10, sigma=500.0, fresh="device"),
        # a smaller, ragged periodic 3-D box, as of a resolution study
        sim("waves", "waves_97x61x75_fp32", nx=97, ny=61, nz=75, steps=20, alpha=0.02, gauss=True),
        # a parameter sweep: uneven shear-layer runs in one handle, spread over streams from graphs as the
        # autotuner sets it
        sim("kh", "kh_sweep_24_fp32", nx=96, ny=384, runs=24, steps=20, alpha=0.02, gauss=True, streams=4, graph=10),
        # a sheet between open faces on the reconnection lattice, monitored: steps, then the conservation numbers
        sim("opensheet", "open_sheet_512_monitor", nx=512, ny=512, steps=20, monitor=True),
        # the learned recovery seed on the benchmark's sheet
        sim("sheet", "learned_sheet_1024_fp32", nx=1024, ny=1024, steps=10, learned=True),
        # training of that seed, resumed: Adam steps on mini-batches of the size the benchmark trains with
        dict(name="mlp_train_1024", kind="train", rows=262144, batch=1024, steps=100),
        # its forward pass over the cells of a large run
        dict(name="mlp_infer_1m", kind="infer", rows=1000003),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _steps(rng, cells, most=60_000_000):
    return max(2, min(_log(rng, 5, 24), most // cells))


def draw(rng):
    what = rng.choice(["1d", "2d", "2d", "2d", "3d", "3d", "sweep", "open", "learned", "train", "grad", "infer"])
    sigma = round(math.exp(rng.uniform(math.log(10.0), math.log(200.0))), 3)
    if what == "1d":
        n = _log(rng, 48, 3000)
        return sim("sheet1d", nx=n, precision="fp64", steps=_log(rng, 40, 400), sigma=sigma, dx=3.0 / n, fresh="host")
    if what == "2d":
        prec = rng.choice(["fp32", "fp32", "fp16", "fp64"])
        side = 512 if prec == "fp64" else 2048
        nx, ny, runs = _log(rng, 24, side), _log(rng, 24, side), rng.choice([1, 1, 2, 3])
        kind = rng.choice(["sheet", "kh", "alfven"])
        streams, graph = rng.choice([(1, 0), (1, 0), (runs, 10)])
        most = 1_500_000 if prec == "fp64" else 60_000_000
        return sim(kind, nx=nx, ny=ny, runs=runs, precision=prec, steps=_steps(rng, nx * ny * runs, most), sigma=sigma,
                   alpha=0.02 if kind == "kh" else 0.1, gauss=kind == "kh", streams=streams, graph=graph)
    if what == "3d":
        kind = rng.choice(["rope", "waves"])
        nx, ny, nz = _log(rng, 20, 200), _log(rng, 20, 200), _log(rng, 20, 200)
        return sim(kind, nx=nx, ny=ny, nz=nz, steps=_steps(rng, nx * ny * nz, 40_000_000),
                   precision=rng.choice(["fp32", "fp32", "fp16"]), sigma=sigma, alpha=0.1 if kind == "rope" else 0.02,
                   gauss=kind == "waves", fresh="device" if kind == "rope" else "")
    if what == "sweep":
        lo = _log(rng, 32, 128)
        runs, hi = rng.randint(4, 24), _log(rng, 128, 512)
        streams, graph = rng.choice([(1, 0), (4, 10)])
        return sim("kh", nx=lo, ny=max(lo, hi), runs=runs, steps=_steps(rng, runs * max(lo, hi) ** 2), sigma=sigma,
                   alpha=0.02, gauss=True, streams=streams, graph=graph)
    if what == "open":
        n = _log(rng, 64, 700)
        return sim("opensheet", nx=n, ny=_log(rng, 64, 700), steps=_steps(rng, n * n), sigma=sigma,
                   precision=rng.choice(["fp32", "fp16"]), monitor=rng.random() < 0.5)
    if what == "learned":
        nx, ny = _log(rng, 64, 1024), _log(rng, 64, 1024)
        return sim("sheet", nx=nx, ny=ny, steps=_steps(rng, nx * ny, 20_000_000), sigma=sigma, learned=True)
    if what == "train":
        return dict(kind="train", rows=_log(rng, 5000, 800_000), batch=_log(rng, 64, 8192), steps=_log(rng, 20, 120))
    if what == "grad":
        return dict(kind="grad", rows=_log(rng, 500, 150_000))
    return dict(kind="infer", rows=_log(rng, 100, 2_000_000))


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _run_specs(case, seed):
    """(nx, ny, nz, sigma, seed) of every run of a handle. Equal runs differ in
    their conductivity; a sweep (kind kh, several runs) has square grids of sides
    nx .. ny."""
    r = np.random.default_rng([seed, 7])
    out = []
    for k in range(case["runs"]):
        nx, ny, sigma = case["nx"], case["ny"], case["sigma"]
        if case["kind"] == "kh" and case["runs"] > 3:
            nx = ny = int(np.random.default_rng([k, nx]).integers(nx, ny + 1))
            sigma = float(10.0 ** r.uniform(1.0, 2.5))
        elif case["runs"] > 1:
            sigma = 10.0 * 10.0 ** k
        out.append((nx, ny, case["nz"], sigma, seed * 1000 + k))
    return out


def _double_tanh(s, length, width):
    return torch.tanh((s + length / 4) / width) - torch.tanh((s - length / 4) / width) - 1.0


def _fields(case, nx, ny, nz, seed, device):
    """Initial n, p (nz, ny, nx), u, B (3, nz, ny, nx), float64."""
    host = np.random.default_rng([seed, nx, ny, nz])
    gen = torch.Generator(device=device)
    gen.manual_seed(seed * 7919 + 13)
    z, y, x = torch.meshgrid(*(torch.arange(k, dtype=torch.float64, device=device) for k in (nz, ny, nx)), indexing="ij")
    one = torch.ones_like(x)
    n, p = one.clone(), one.clone()
    u, B = torch.zeros((3,) + x.shape, dtype=torch.float64, device=device), torch.zeros((3,) + x.shape, dtype=torch.float64, device=device)
    a, ph = host.uniform(0.9, 1.1, 8), host.uniform(0.0, 2 * math.pi, 8)
    kind = case["kind"]
    if kind == "sheet":  # periodic double current sheet along y
        s = torch.remainder(x + 0.5 + nx * ph[0] / (2 * math.pi), nx) - nx / 2
        B[1] = 0.1 * a[0] * _double_tanh(s, float(nx), 8.0 * a[1])
    elif kind == "sheet1d":  # the paper's sheet on [-1.5, 1.5] at t0 = 1
        p = 50.0 * a[0] * one
        B[1] = a[1] * torch.erf(0.5 * math.sqrt(case["sigma"]) * (-1.5 + (x + 0.5) * case["dx"]))
    elif kind == "alfven":  # one wavelength along x, small amplitude
        k, amp, B0 = 2 * math.pi / nx, 1e-3 * a[0], 0.1
        B[0], B[2] = B0, amp * torch.sin(k * (x + 0.5) + ph[0])
        u[2] = -B[2] / math.sqrt(5.0 + B0 * B0)
    elif kind == "kh":  # two shear layers along x with a reversed field and noise
        s = y + 0.5 - ny / 2
        prof = _double_tanh(s, float(ny), 2.0)
        d = torch.minimum((s + ny / 4).abs(), (s - ny / 4).abs())
        noise = torch.rand(x.shape, dtype=torch.float64, device=device, generator=gen) * 2 - 1
        u[0], u[1], B[0] = 0.1 * a[0] * prof, 1e-3 * noise * torch.exp(-(d * d) / 100.0), 0.1 * a[1] * prof
    elif kind == "opensheet":  # one layer across the middle, open x faces
        B[1] = 0.1 * a[0] * torch.tanh((x + 0.5 - nx * (0.5 + 0.02 * math.sin(ph[0]))) / (8.0 * a[1]))
    elif kind == "waves":  # a magnetised box with a few smooth modes
        kx, ky, kz = (2 * math.pi / m for m in (nx, ny, nz))
        n = 1.0 + 0.05 * a[0] * torch.sin(kx * x + ky * y + ph[0])
        u[0] = 0.02 * a[1] * torch.sin(ky * y + ph[1]) * torch.cos(kz * z + ph[2])
        u[1] = 0.02 * a[2] * torch.sin(kz * z + ph[3])
        u[2] = 0.02 * a[3] * torch.sin(kx * x + ph[4])
        B[0], B[1], B[2] = 0.05 * torch.sin(kz * z + ph[5]), 0.05 * torch.sin(kx * x + ph[6]), 0.05 * a[4]
    elif kind == "rope":  # arched flux rope over [-3, 3]^2 x [0, 6]: four line currents, an image, a rope of radius r0
        X, Z = -3.0 + (x + 0.5) * 6.0 / nx, (z + 0.5) * 6.0 / nz
        r0, h, cb = 0.5, 2.0 * a[0], 0.2534 * a[1]
        gx, gz = torch.zeros_like(X), torch.zeros_like(X)
        for xc, zc, w in ((-0.3, -0.3, cb), (0.3, -0.3, cb), (-1.5, -0.3, -cb), (1.5, -0.3, -cb), (0.0, -h, -0.5 * r0)):
            q = (X - xc) ** 2 + (Z - zc) ** 2
            gx += w * 2 * (X - xc) / q
            gz += w * 2 * (Z - zc) / q
        r = torch.sqrt(X * X + (Z - h) ** 2).clamp_min(1e-300)
        dl = torch.where(r <= r0, r / r0, r0 / r) / r
        gx += dl * X
        gz += dl * (Z - h)
        top = torch.sqrt((gx * gx + gz * gz).max())
        B[0], B[2] = -gz * (0.05 / top), gx * (0.05 / top)
        B[1] = torch.where(r <= r0, 0.2 * torch.sqrt((1.0 - (r / r0) ** 2).clamp_min(0.0)), torch.zeros_like(r))
    else:
        raise ValueError(kind)
    return n, p, u, B


def _faces(case):
    if case["kind"] in ("sheet1d", "opensheet"):
        return (L.OPEN, L.OPEN, L.PERIODIC, L.PERIODIC, L.PERIODIC, L.PERIODIC)
    if case["kind"] == "rope":
        return (L.OPEN,) * 4 + (L.DRIVEN, L.OPEN)
    return (L.PERIODIC,) * 6


def _drive(case):
    """Speed and thickness of the driven layers (the paper's 0.2343 of a 6-high box)."""
    return (0.05, int(math.ceil(0.2343 / 6.0 * case["nz"]))) if case["kind"] == "rope" else (0.0, 0)


def _network(seed, device):
    """float32 parameters of a network that carries T^{0a}/T^00 through its ReLU
    layers to beta ~ 0.8 T^{0a}/T^00 (n = p = 1), among small random weights: as
    good a guess as a trained one gives."""
    r = np.random.default_rng([seed, 3])
    shapes = ((64, 20), (64, 64), (64, 64), (4, 64))
    W = [r.normal(0.0, 1e-3, s) for s in shapes]
    for a in range(3):
        W[0][2 * a, a], W[0][2 * a + 1, a] = 1.0, -1.0
        W[3][a, 2 * a], W[3][a, 2 * a + 1] = 0.8, -0.8
    for k in (1, 2):
        for j in range(6):
            W[k][j, j] = 1.0
    parts = []
    for w in W:
        parts += [w.reshape(-1), r.normal(0.0, 1e-4, w.shape[0])]
    return torch.tensor(np.concatenate(parts), dtype=torch.float32, device=device)


def _initial_network(seed, device):
    """He-initialised float32 parameters, as a training starts from."""
    r = np.random.default_rng([seed, 5])
    parts = []
    for o, k, s in ((64, 20, 1.0), (64, 64, 1.0), (64, 64, 1.0), (4, 64, 0.1)):
        parts += [r.normal(0.0, s * math.sqrt(2.0 / k), o * k), np.zeros(o)]
    return torch.tensor(np.concatenate(parts), dtype=torch.float32, device=device)


def _adam(seed, device):
    """Adam's moments as a resumed training has them: first ~ 0, second of an earlier, rougher stage."""
    v = 10.0 ** np.random.default_rng([seed, 11]).uniform(-4.0, -2.0, L.MLP_NPARAM)
    return torch.tensor(np.concatenate([np.zeros(L.MLP_NPARAM), v]), dtype=torch.float32, device=device)


def _samples(rows, seed, device):
    """Training rows of cells of a magnetised flow: the normalised moments of a
    perfect fluid with fields (20), then beta and eps / T^00 - 1."""
    gen = torch.Generator(device=device)
    gen.manual_seed(seed * 31 + 17)
    v = torch.rand((12, rows), dtype=torch.float64, device=device, generator=gen)
    b = (v[0:3] * 2 - 1) * 0.3
    n, p = 0.2 + 1.8 * v[3], 0.9 + 0.2 * v[4]
    B, E0 = (v[5:8] * 2 - 1) * 0.1, (v[8:11] * 2 - 1) * 1e-3
    E = -torch.linalg.cross(b, B, dim=0) + E0
    eps = n + p / (GAMMA_AD - 1.0)
    g2 = 1.0 / (1.0 - (b * b).sum(0))
    w = (eps + p) * g2
    em = 0.5 * ((E * E).sum(0) + (B * B).sum(0))
    S = torch.linalg.cross(E, B, dim=0)
    T00 = w - p + em
    T0a = w * b + S
    T = [w * b[i] * b[j] + (p + em if i == j else 0.0) - E[i] * E[j] - B[i] * B[j]
         for i, j in ((0, 0), (1, 1), (2, 2), (0, 1), (0, 2), (1, 2))]
    out = torch.empty((rows, 24), dtype=torch.float64, device=device)
    out[:, 0:3] = (T0a / T00).T
    for m in range(6):
        out[:, 3 + m] = T[m] / T00
    out[:, 9:12] = b.T
    out[:, 12] = n * torch.sqrt(g2) / T00
    out[:, 13:16], out[:, 16:19] = (E / torch.sqrt(T00)).T, (B / torch.sqrt(T00)).T
    out[:, 19] = 1.0
    out[:, 20:23], out[:, 23] = b.T, eps / T00 - 1.0
    return out.float()


def prepare(case, seed):
    dev = "cuda"
    if case["kind"] in ("train", "grad", "infer"):
        data = _samples(case["rows"], seed, dev)
        if case["kind"] == "infer":
            return {"case": case, "blob": L.mlp_pack(_network(seed, dev)), "features": data[:, :20].contiguous()}
        return {"case": case, "data": data, "params": _initial_network(seed, dev), "seed": seed,
                "adam": _adam(seed, dev)}
    specs = _run_specs(case, seed)
    u0, layers = _drive(case)
    params = [L.make_params(nx, ny, nz, bc=_faces(case), tau=TAU, sigma=sigma, gamma_ad=GAMMA_AD, alpha=case["alpha"],
                            c=case["c"], dx=case["dx"], drive_u0=u0, drive_layers=layers,
                            precision=PRECISION[case["precision"]],
                            recovery=L.RECOVERY_MLP if case["learned"] else L.RECOVERY_PLAIN,
                            flags=L.FLAG_GAUSS_CHARGE if case["gauss"] else 0)
              for nx, ny, nz, sigma, _ in specs]
    solver = L.Solver(params, stream=torch.cuda.current_stream())
    if case["learned"]:
        solver.set_mlp_weights(_network(seed, dev))
    if case["streams"] > 1 or case["graph"]:
        solver.set_schedule(kind=L.SCHED_PER_RUN, streams=case["streams"], graph_steps=case["graph"])
    first = []
    for r, (nx, ny, nz, _, s) in enumerate(specs):
        f = [t.contiguous() for t in _fields(case, nx, ny, nz, s, dev)]
        if case["fresh"]:
            first.append([t.cpu().numpy() for t in f] if case["fresh"] == "host" else f)
        else:
            solver.init_fields_device(r, *f)
    moments = [torch.empty((L.NMOMENTS, n), dtype=torch.float64, device=dev) for n in solver.cells]
    torch.cuda.synchronize()
    return {"case": case, "solver": solver, "first": first, "moments": moments}


def run(state):
    case = state["case"]
    if case["kind"] == "train":
        loss = L.mlp_train(state["params"], state["adam"], state["data"], case["steps"], case["batch"], 1e-3,
                           seed=state["seed"])
        return {"params": state["params"], "adam": state["adam"], "loss": loss}
    if case["kind"] == "grad":
        loss, grad = L.mlp_grad(state["params"], state["data"])
        return {"loss": torch.tensor([loss], dtype=torch.float32), "grad": grad}
    if case["kind"] == "infer":
        return {"out": L.mlp_infer(state["blob"], state["features"])}
    solver, out = state["solver"], []
    for r, f in enumerate(state["first"]):
        (solver.init_fields if case["fresh"] == "host" else solver.init_fields_device)(r, *f)
    solver.step(case["steps"])
    for r, m in enumerate(state["moments"]):
        solver.moments_device(r, m)
        snap = m.to(SNAPSHOT[case["precision"]])
        out.append({"fluid": snap[:6], "em": snap[6:]})
    if case["monitor"]:
        out.append([torch.from_numpy(solver.diagnostics(r)).to(SNAPSHOT[case["precision"]]) for r in range(case["runs"])])
    return out


def work(case):
    if case["kind"] == "train":
        each = case["batch"] * case["steps"]
        return {"bytes": each * 96 + case["steps"] * 7 * 4 * L.MLP_NPARAM, "flops": each * 6.0 * L.MLP_NPARAM}
    if case["kind"] == "grad":
        return {"bytes": case["rows"] * 96 + 8 * L.MLP_NPARAM, "flops": case["rows"] * 6.0 * L.MLP_NPARAM}
    if case["kind"] == "infer":
        return {"bytes": case["rows"] * 96, "flops": case["rows"] * 2.0 * L.MLP_NPARAM}
    cells = sum(nx * ny * nz for nx, ny, nz, _, _ in _run_specs(case, 0))
    size = {"fp64": 8, "fp32": 4, "fp16": 2}[case["precision"]]
    prim = 96 if case["precision"] == "fp64" else 48
    dim = 3 if case["nz"] > 1 else 2 if case["ny"] > 1 else 1
    extra = cells * (prim + 16 * size)  # the snapshot
    if case["monitor"]:
        extra += cells * BYTES_PER_UPDATE[case["precision"]] // 2
    if case["fresh"]:
        extra += cells * (64 + BYTES_PER_UPDATE[case["precision"]] // 2)
    return {"bytes": case["steps"] * cells * BYTES_PER_UPDATE[case["precision"]] + extra,
            "flops": float(case["steps"] * cells * FLOPS_PER_UPDATE[dim] * (1.0 if not case["learned"] else 11.0))}


# ---------------------------------------------------------------------------
# the method in float64
# ---------------------------------------------------------------------------
_C = [(0, 0, 0)] + [tuple(s * (k == a) for k in range(3)) for a in range(3) for s in (1, -1)]
for _a, _b in ((0, 1), (0, 2), (1, 2)):
    for _s, _t in ((1, 1), (-1, -1), (1, -1), (-1, 1)):
        _C.append(tuple(_s * (k == _a) + _t * (k == _b) for k in range(3)))
_PAIRS = ((0, 0), (1, 1), (2, 2), (0, 1), (0, 2), (1, 2))
_PLANES = ((0, 1, 2, 1.0), (0, 2, 1, -1.0), (1, 2, 0, 1.0))  # axes, normal, orientation
_HOPS = ((1, 1), (-1, 1), (-1, -1), (1, -1))
_Q = math.sqrt(19.0 / 27.0)


def _cross(a, b):
    return torch.stack((a[1] * b[2] - a[2] * b[1], a[2] * b[0] - a[0] * b[2], a[0] * b[1] - a[1] * b[0]))


def _mul(M, v):
    """Matrix (rows x k) times a stack of k fields."""
    return (M @ v.reshape(v.shape[0], -1)).reshape((M.shape[0],) + v.shape[1:])


class _Exact:
    def __init__(self, case, nx, ny, nz, sigma, seed, device):
        self.shape, self.dev, self.sigma = (nz, ny, nx), device, sigma
        self.c, self.dx, self.gauss = case["c"], case["dx"], case["gauss"]
        self.dt = self.dx / (math.sqrt(2.0) * self.c)
        self.courant = _Q * self.c * self.dt / self.dx
        self.visc = case["alpha"] * self.c * self.dt / self.dx
        self.gm1 = GAMMA_AD - 1.0
        self.eps0 = 1.0 / self.c ** 2
        f = _faces(case)
        self.open = [f[2 * a] != L.PERIODIC for a in range(3)]
        self.u0, self.layers = _drive(case)
        self._tables()
        n, p, u, B = _fields(case, nx, ny, nz, seed, device)
        E = -_cross(u, B)
        self.n, self.eps, self.u, self.B, self.E = n, n * self.c ** 2 + p / self.gm1, u, B, E
        self.rho = self.eps0 * self.div(E)
        if self.layers:
            X = -3.0 + (torch.arange(nx, dtype=torch.float64, device=device) + 0.5) * 6.0 / nx
            Y = (-3.0 + (torch.arange(ny, dtype=torch.float64, device=device) + 0.5) * 6.0 / ny)[:, None]
            xs = torch.where(X < 0, X, X - 3.0)
            self.drive = torch.stack((self.u0 * torch.sin(math.pi * xs / 3) * torch.cos(math.pi * Y / 6),
                                      self.u0 * torch.cos(math.pi * xs / 3) * torch.sin(math.pi * Y / 6),
                                      torch.zeros_like(Y * X)))[:, None]
        self.f = self.feq(self.n, self.eps, self.u, self.E, self.B)
        self.g = self.geq(self.n, self.u)
        # the mean initial field's share of T^00 and T^0a, which the library's diagnostics leave out
        self.field = [0.5 * self.eps0 * float((E * E + self.c ** 2 * B * B).sum())]
        self.field += [-self.eps0 * self.c * float(v.sum()) for v in _cross(B, E)]
        self.h = self.heq(self.E, self.B, self.ohm(self.E, self.u, self.B, self.rho), self.rho)

    def _tables(self):
        t = lambda m: torch.tensor(m, dtype=torch.float64, device=self.dev)  # noqa: E731
        w = [(-44.0 / 361.0, 99.0 / 722.0, 9.0 / 361.0)[sum(map(abs, c))] for c in _C]
        wg = [(0.1, 6.0 / 95.0, 33.0 / 760.0)[sum(map(abs, c))] for c in _C]
        l1 = math.sqrt(19.0) * (math.sqrt(27.0) / 2 - 1) / (0.375 * (9 - 2 * math.sqrt(3.0)))
        # feq on (p, eps, W b (3), W b_a b_b (6), Y (3), X (6)), W = (eps + p) gamma^2
        F = []
        for i, c in enumerate(_C):
            rest = 0.75 * 361.0 / 33.0 if i == 0 else 0.0
            row = [3.0 + 3.0 * rest, -rest] + [0.75 * l1 * c[a] for a in range(3)]
            for a, b in _PAIRS:
                row.append(0.75 * (4.0 / 15.0) * (19.0 * c[a] ** 2 - 4.0) if a == b else 0.75 * 19.0 * c[a] * c[b])
            row += [-math.sqrt(19.0 / 3.0) * c[a] for a in range(3)]
            for a, b in _PAIRS:
                row.append(2.3 - 3.8 * c[a] ** 2 if a == b else -14.25 * c[a] * c[b])
            F.append([w[i] * v for v in row])
        self.F = t(F)
        # geq on n gamma (1, b (3), b_a b_b (6))
        self.G = t([[wg[i]] + [wg[i] * 3 * _Q * c[a] for a in range(3)] +
                    [wg[i] * (4.5 * _Q ** 2 * c[a] ** 2 - 1.5 if a == b else 9 * _Q ** 2 * c[a] * c[b]) for a, b in _PAIRS]
                    for i, c in enumerate(_C)])
        self.T = t([[1.0] * 19] + [[_Q * c[a] for c in _C] for a in range(3)] +
                   [[_Q ** 2 * c[a] * c[b] for c in _C] for a, b in _PAIRS])
        self.chat = t(_C)
        v, e, b = [], [], []
        for a1, a2, nrm, o in _PLANES:
            for i in range(4):
                for j in range(2):
                    vv, ee, bb = [0.0] * 3, [0.0] * 3, [0.0] * 3
                    vv[a1], vv[a2] = _HOPS[i]
                    sg = 1.0 if j == 0 else -1.0
                    ee[a1], ee[a2] = (sg * s for s in _HOPS[(i + 3) % 4])
                    bb[nrm] = -sg * o
                    v.append(vv), e.append(ee), b.append(bb)
        self.hops, r2 = [[int(k) for k in vv] for vv in v], math.sqrt(2.0)
        self.He, self.Hb = t(e) * (r2 / 2 * self.c), t(b)
        # heq on (J, E, B), k = 0..23
        self.H = torch.cat((t(v) * (r2 * self.c / 16), self.He / (8 * self.c ** 2), self.Hb / 8), 1)

    # stencil access: wrapped on a periodic axis, clamped on an open one (axis 0 = x, the last dimension)
    def at(self, a, axis, d):
        if d == 0:
            return a
        dim, m = a.dim() - 1 - axis, a.shape[a.dim() - 1 - axis]
        if not self.open[axis]:
            return torch.roll(a, -d, dim)
        return a.index_select(dim, (torch.arange(m, device=a.device) + d).clamp(0, m - 1))

    def div(self, E):
        s = torch.zeros(self.shape, dtype=torch.float64, device=self.dev)
        for a in range(3):
            if self.shape[2 - a] > 1:
                s = s + (self.at(E[a], a, 1) - self.at(E[a], a, -1)) / (2 * self.dx)
        return s

    def feq(self, n, eps, u, E, B):
        b, p = u / self.c, self.gm1 * (eps - n * self.c ** 2)
        W = (eps + p) / (1.0 - (b * b).sum(0))
        X = [self.eps0 * (E[i] * E[j] + self.c ** 2 * B[i] * B[j]) for i, j in _PAIRS]
        Y = self.eps0 * self.c * _cross(B, E)
        return _mul(self.F, torch.stack([p, eps] + [W * b[a] for a in range(3)] + [W * b[i] * b[j] for i, j in _PAIRS] +
                                        list(Y) + X))

    def geq(self, n, u):
        b = u / self.c
        ng = n / torch.sqrt(1.0 - (b * b).sum(0))
        return _mul(self.G, torch.stack([ng] + [ng * b[a] for a in range(3)] + [ng * b[i] * b[j] for i, j in _PAIRS]))

    def heq(self, E, B, J, rho):
        return torch.cat((_mul(self.H, torch.cat((J, E, B))), rho[None]))

    def ohm(self, E, u, B, rho):
        g = 1.0 / torch.sqrt(1.0 - (u * u).sum(0) / self.c ** 2)
        return self.sigma * g * (E + _cross(u, B) - (E * u).sum(0) * u / self.c ** 2) + rho * u

    def stream(self, f, visc):
        """One flux-limited step of every population (dimension 0)."""
        kap = 0.5 * (1.0 - self.courant)

        def limited(a, b):
            return torch.where(a * b > 0, torch.where(a.abs() < b.abs(), a, b), torch.zeros_like(a))

        out = f.clone()
        for a in range(3):
            if self.shape[2 - a] == 1:
                continue  # every neighbour is the cell itself
            for s in (1, -1):
                idx = [i for i, c in enumerate(_C) if c[a] == s]
                v = f[idx]
                m2, m1, p1 = (self.at(v, a, k * s) for k in (-2, -1, 1))
                d0 = v - m1
                out[idx] -= self.courant * (d0 + kap * (limited(p1 - v, d0) - limited(d0, m1 - m2)))
            if visc:
                out[1:] += self.visc * (self.at(f[1:], a, 1) + self.at(f[1:], a, -1) - 2 * f[1:])
        return out

    def recover(self, f, g, h, rho_j):
        c, e0 = self.c, self.eps0
        T = _mul(self.T, f)
        N0 = g.sum(0)
        Ep, B = _mul(self.He.T.contiguous(), h[:24]), _mul(self.Hb.T.contiguous(), h[:24])
        hs = 0.5 * self.dt * c * c * self.sigma
        B2 = (B * B).sum(0)
        E, b = self.E.clone(), self.u / c
        p = self.gm1 * (self.eps - self.n * c * c)
        best, worse = math.inf, 0
        for outer in range(80):
            E2, ExB = (E * E).sum(0), _cross(E, B)
            a00 = T[0] - e0 * E2
            a0 = T[1:4] - e0 * c * ExB
            s = 0.5 * e0 * (c * c * B2 - E2)
            A = {}
            for m, (i, j) in enumerate(_PAIRS):
                A[i, j] = A[j, i] = T[4 + m] + e0 * E[i] * E[j] - e0 * c * c * ((B2 if i == j else 0.0) - B[i] * B[j])
            shift = p - s
            for _ in range(3):
                w0 = a00 + shift - (a0 * b).sum(0)
                b = torch.stack([a0[i] + shift * b[i] - (A[i, 0] * b[0] + A[i, 1] * b[1] + A[i, 2] * b[2])
                                 for i in range(3)]) / w0
            lam = a00 - (a0 * b).sum(0)
            g2 = 1.0 / (1.0 - (b * b).sum(0))
            gam, u = torch.sqrt(g2), c * b
            k = hs * gam
            rhs = Ep - k * _cross(u, B) - 0.5 * self.dt * c * c * rho_j * u
            En = (rhs + (k / (c * c)) * (u * rhs).sum(0) / (1.0 + k / g2) * u) / (1.0 + k)
            eps, n = lam - s, N0 / gam
            p = self.gm1 * (eps - n * c * c)
            d = float((En - E).abs().max())
            if d >= best:
                worse += 1
            best = min(best, d)
            if d <= 1e-16 * float(En.abs().max() + c * B.abs().max()) or worse >= 3:
                break
            r = B2 * (k / (1.0 + k)) / ((eps + p) * g2)
            dE = En - E
            par = (dE * B).sum(0) / B2.clamp_min(1e-300) * B  # the part along B does not feed back
            E = E + par + (dE - par) / (1.0 + r)
        J = (Ep - En) / (0.5 * self.dt * c * c)
        return n, eps, u, En, B, h.sum(0), J

    def step(self):
        c = self.c
        f, g = self.stream(self.f, True), self.stream(self.g, False)
        h = torch.empty_like(self.h)
        for k in range(24):
            v = self.h[k]
            for a in range(3):
                v = self.at(v, a, -self.hops[k][a]) if self.shape[2 - a] > 1 else v
            h[k] = v
        h[24] = self.h[24]
        rho = h.sum(0)
        rho_j = self.eps0 * self.div(self.E) if self.gauss else rho
        self.n, self.eps, self.u, self.E, self.B, self.rho, J = self.recover(f, g, h, rho_j)
        b = self.u / c
        gam = 1.0 / torch.sqrt(1.0 - (b * b).sum(0))
        K = gam / TAU * (1.0 - _Q * _mul(self.chat, b))
        self.f = f - K * (f - self.feq(self.n, self.eps, self.u, self.E, self.B))
        self.g = g - (g - self.geq(self.n, self.u)) / TAU
        self.h = 2 * self.heq(self.E, self.B, J, self.rho) - h
        self.boundaries()

    def boundaries(self):
        for a in range(3):
            m = self.shape[2 - a]
            if self.open[a] and m >= 3:  # open faces copy their interior neighbour
                idx = torch.arange(m, device=self.dev).clamp(1, m - 2)
                for name in ("f", "g", "h", "n", "eps", "u", "E", "B", "rho"):
                    v = getattr(self, name)
                    setattr(self, name, v.index_select(v.dim() - 1 - a, idx))
        for a in range(3):
            m = self.shape[2 - a]
            if self.open[a] and m >= 3:
                for s, at in ((1, 0), (-1, m - 1)):
                    self.normal_field(a, s, at)
        if self.layers:  # the driven bottom: two vortices, ideal field, equilibrium
            lo = slice(0, self.layers)
            n, eps, B, rho = self.n[lo], self.eps[lo], self.B[:, lo], self.rho[lo]
            u = self.drive.expand_as(B).contiguous()
            E = -_cross(u, B)
            self.u[:, lo], self.E[:, lo] = u, E
            self.f[:, lo], self.g[:, lo] = self.feq(n, eps, u, E, B), self.geq(n, u)
            self.h[:, lo] = self.heq(E, B, self.ohm(E, u, B, rho), rho)

    def normal_field(self, a, s, at):
        """B along axis a on one open face, so that div B of the first interior layer vanishes."""
        dim = 2 - a
        layer = lambda v, k: v.narrow(v.dim() - 1 - a, k, 1)  # noqa: E731
        tang = torch.zeros_like(layer(self.B[a], at))
        for t in range(3):
            if t != a and self.shape[2 - t] > 1:
                Bt = layer(self.B[t], at + s)
                tang = tang + (self.at(Bt, t, 1) - self.at(Bt, t, -1)) / (2 * self.dx)
        new = layer(self.B[a], at + 2 * s) + s * 2 * self.dx * tang
        n, eps, u, E, B = (layer(v, at) for v in (self.n, self.eps, self.u, self.E, self.B))
        Bn = B.clone()
        Bn[a] = new
        dB, b = new - B[a], u / self.c
        K = (1.0 - _Q * _mul(self.chat, b)) / (TAU * torch.sqrt(1.0 - (b * b).sum(0)))
        f, h = layer(self.f, at), layer(self.h, at)
        f += K * (self.feq(n, eps, u, E, Bn) - self.feq(n, eps, u, E, B))
        h[:24] += (self.Hb[:, a].reshape(-1, 1, 1, 1) / 8) * dB
        self.B[a].narrow(dim, at, 1).copy_(new)

    def moments(self):
        J = self.ohm(self.E, self.u, self.B, self.rho)
        p = self.gm1 * (self.eps - self.n * self.c ** 2)
        m = torch.cat((self.n[None], p[None], self.eps[None], self.u, self.E, self.B, self.rho[None], J))
        return m.reshape(16, -1)

    def diagnostics(self):
        div = self.div(self.B)
        cells = div.numel()
        T = [float(self.f.sum())] + [_Q * float((self.chat[:, a].reshape(-1, 1, 1, 1) * self.f).sum()) for a in range(3)]
        return torch.tensor([float(self.g.sum())] + [t - e for t, e in zip(T, self.field)] +
                            [float(self.h.sum()), float(div.abs().max()), math.sqrt(float((div * div).sum()) / cells), 0.0,
                             float(cells)], dtype=torch.float64)


def _forward64(P, X):
    """Activations of the 20-64-64-64-4 network in float64."""
    W, o = [], 0
    for k, i in ((64, 20), (64, 64), (64, 64), (4, 64)):
        W.append((P[o:o + k * i].reshape(k, i), P[o + k * i:o + k * i + k]))
        o += k * i + k
    acts = [X]
    for j, (w, b) in enumerate(W):
        v = acts[-1] @ w.T + b
        acts.append(v.clamp_min(0.0) if j < 3 else v)
    return W, acts


def _grad64(P, rows):
    W, acts = _forward64(P, rows[:, :20])
    e = acts[-1] - rows[:, 20:]
    d, parts = 2.0 * e / rows.shape[0], []
    for j in (3, 2, 1, 0):
        parts = [(d.T @ acts[j]).reshape(-1), d.sum(0)] + parts
        if j:
            d = (d @ W[j][0]) * (acts[j] > 0)
    return (e * e).sum() / rows.shape[0], torch.cat(parts)


def _splitmix64(x):
    with np.errstate(over="ignore"):
        x = np.asarray(x, dtype=np.uint64) + np.uint64(0x9E3779B97F4A7C15)
        x = (x ^ (x >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        x = (x ^ (x >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
        return x ^ (x >> np.uint64(31))


def _train64(case, seed, device):
    """The documented training: rows drawn by a hash of (seed, step, j), Adam."""
    P = _initial_network(seed, device).double()
    data = _samples(case["rows"], seed, device).double()
    m, v = _adam(seed, device).double().reshape(2, -1)
    # the betas are the float32 values of 0.9 and 0.999
    b1, b2, losses = float(np.float32(0.9)), float(np.float32(0.999)), []
    lr, tiny = float(np.float32(1e-3)), float(np.float32(1e-8))
    with np.errstate(over="ignore"):
        for t in range(case["steps"]):
            key = _splitmix64(np.uint64(seed) + np.uint64(t + 1)) | np.uint64(1)
            j = np.arange(case["batch"], dtype=np.uint64) * np.uint64(0x2545F4914F6CDD1D)
            rows = (_splitmix64(key ^ j) % np.uint64(case["rows"])).astype(np.int64)
            loss, g = _grad64(P, data[torch.from_numpy(rows).to(device)])
            losses.append(loss)
            m, v = b1 * m + (1 - b1) * g, b2 * v + (1 - b2) * g * g
            P = P - lr * (m / (1 - b1 ** (t + 1))) / (torch.sqrt(v / (1 - b2 ** (t + 1))) + tiny)
    return {"params": P, "adam": torch.cat((m, v)), "loss": torch.stack(losses)}


def exact(case, seed):
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    if case["kind"] == "train":
        return _train64(case, seed, dev)
    if case["kind"] == "grad":
        loss, grad = _grad64(_initial_network(seed, dev).double(), _samples(case["rows"], seed, dev).double())
        return {"loss": loss.reshape(1), "grad": grad}
    if case["kind"] == "infer":
        return {"out": _forward64(_network(seed, dev).double(), _samples(case["rows"], seed, dev)[:, :20].double())[1][-1]}
    specs = _run_specs(case, seed)
    cells = sum(nx * ny * nz for nx, ny, nz, _, _ in specs)
    if case["steps"] * (cells * 2.4e-8 + 0.016 * case["runs"]) > 18.0:
        return None
    small = dev if cells > 4000 else "cpu"  # short arrays: the host's launches are the shorter ones
    out, diag = [], []
    for nx, ny, nz, sigma, s in specs:
        sm = _Exact(case, nx, ny, nz, sigma, s, small)
        for _ in range(case["steps"]):
            sm.step()
        m = sm.moments()
        out.append({"fluid": m[:6], "em": m[6:]})
        if case["monitor"]:
            diag.append(sm.diagnostics())
    return out + ([diag] if case["monitor"] else [])
