"""The work a user of this package has it do, as timed cases.

Each case is one call (or the few calls that belong together) through the package's public entry
points, on the sizes of the package's own configurations, tests and benchmark, and on odd and
ragged sizes of the same range:

  step    Solver.step from an initial state: 1D, 2D and 3D, FP32 and FP64
  batch   BatchSolver.step: many uneven 2D grids advanced together
  wave    wave_run: the linear-wave example with its energy after each step
  audit   what a program writes out beside its steps: cfl_dt, totals and primitive planes
  host    Solver.step_host: the state in from pinned host memory, steps, the state back
  train   MLP.train: the tuner's cost model fitted to its records

Times and dt of FP32 runs carry the accuracy of the FP32 signal they come from and are returned
as float32; those of FP64 runs as float64.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1204_4779_gb300 import costmodel, hydro

DTYPES = {"f32": torch.float32, "f64": torch.float64}


def listed():
    return [
        # The plain method's first problem: Sod's tube on 1024 cells to t = 0.2 with outflow ends.
        # Some thousand steps of a grid that fits one SM: latency and launches are all there is.
        {"name": "sod1d_f64", "kind": "step", "flow": "sod", "dtype": "f64", "dim": 1, "nx": 1024,
         "ny": 1, "nz": 1, "bc": "o", "steps": 100000, "t_end": 0.2},
        # The 2D shear layer of the benchmark's second configuration, 100 steps in FP32.
        {"name": "shear2d_f32", "kind": "step", "flow": "shear", "dtype": "f32", "dim": 2,
         "nx": 1024, "ny": 1024, "nz": 1, "bc": "pp", "steps": 100, "t_end": 0.0},
        # The same layer in FP64, the form whose result is the reference.
        {"name": "shear2d_f64", "kind": "step", "flow": "shear", "dtype": "f64", "dim": 2,
         "nx": 1024, "ny": 1024, "nz": 1, "bc": "pp", "steps": 20, "t_end": 0.0},
        # A larger 2D grid of odd sides with open boundaries across the layer.
        {"name": "shear2d_ragged_f32", "kind": "step", "flow": "shear", "dtype": "f32", "dim": 2,
         "nx": 3001, "ny": 2003, "nz": 1, "bc": "po", "steps": 20, "t_end": 0.0},
        # The 3D blast at the small tuning size: an ordinary 3D run that does not fill many waves.
        {"name": "blast3d_128_f32", "kind": "step", "flow": "blast", "dtype": "f32", "dim": 3,
         "nx": 128, "ny": 128, "nz": 128, "bc": "ppp", "steps": 50, "t_end": 0.0},
        # The headline: the 3D blast on 512^3.
        {"name": "blast3d_512_f32", "kind": "step", "flow": "blast", "dtype": "f32", "dim": 3,
         "nx": 512, "ny": 512, "nz": 512, "bc": "ppp", "steps": 10, "t_end": 0.0},
        # A 3D FP64 run of odd sides with open ends along z.
        {"name": "blast3d_ragged_f64", "kind": "step", "flow": "blast", "dtype": "f64", "dim": 3,
         "nx": 97, "ny": 83, "nz": 75, "bc": "ppo", "steps": 20, "t_end": 0.0},
        # The batched configuration: 4096 grids with sides drawn log-uniformly from 32 to 512.
        {"name": "batch4096_f32", "kind": "batch", "dtype": "f32", "grids": 4096, "lo": 32,
         "hi": 512, "steps": 10},
        # The linear-wave example at the upper end of the paper's range of N.
        {"name": "wave3072_f64", "kind": "wave", "dtype": "f64", "n": 3072, "steps": 300},
        # What a run writes out: the stable dt, the conserved totals and the primitive planes of
        # the headline's state.
        {"name": "audit512_f32", "kind": "audit", "dtype": "f32", "nx": 512, "ny": 512, "nz": 512},
        # A state kept in host memory and advanced through the GPU.
        {"name": "host3d_256_f32", "kind": "host", "dtype": "f32", "nx": 256, "ny": 256, "nz": 256,
         "steps": 5},
        # The tuner's cost model retrained on its full set of records.
        {"name": "train4200", "kind": "train", "records": 4200, "features": 35, "hidden": 64,
         "epochs": 200},
    ]


def _log(rng, lo, hi):
    """An integer drawn log-uniformly from [lo, hi]."""
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _bc(rng, dim):
    return "".join(rng.choice("ppo") for _ in range(dim))


def draw(rng):
    kind = rng.choice(["step1", "step2", "step2", "step3", "step3", "batch", "wave", "audit",
                       "host", "train"])
    if kind == "step1":
        dtype = rng.choice(["f64", "f32"])
        return {"kind": "step", "flow": rng.choice(["sod", "smooth"]), "dtype": dtype, "dim": 1,
                "nx": _log(rng, 64, 200000), "ny": 1, "nz": 1, "bc": _bc(rng, 1),
                "steps": _log(rng, 10, 300), "t_end": 0.0}
    if kind == "step2":
        dtype = rng.choice(["f32", "f32", "f64"])
        nx, ny = (_log(rng, 32, 4096 if dtype == "f32" else 1024) for _ in range(2))
        most = (5e8 if dtype == "f32" else 2e7) / (nx * ny)
        return {"kind": "step", "flow": rng.choice(["shear", "smooth"]), "dtype": dtype, "dim": 2,
                "nx": nx, "ny": ny, "nz": 1, "bc": _bc(rng, 2),
                "steps": _log(rng, 5, max(6, min(100, int(most)))), "t_end": 0.0}
    if kind == "step3":
        dtype = rng.choice(["f32", "f32", "f32", "f64"])
        nx, ny, nz = (_log(rng, 16, 384 if dtype == "f32" else 128) for _ in range(3))
        most = (5e8 if dtype == "f32" else 1e7) / (nx * ny * nz)
        return {"kind": "step", "flow": rng.choice(["blast", "smooth"]), "dtype": dtype, "dim": 3,
                "nx": nx, "ny": ny, "nz": nz, "bc": _bc(rng, 3),
                "steps": _log(rng, 4, max(5, min(60, int(most)))), "t_end": 0.0}
    if kind == "batch":
        lo = _log(rng, 16, 64)
        return {"kind": "batch", "dtype": "f32", "grids": _log(rng, 16, 2048), "lo": lo,
                "hi": _log(rng, 2 * lo, 512), "steps": rng.randint(5, 10)}
    if kind == "wave":
        # FP32 resolves the second differences of a smooth wave on small grids only
        dtype = rng.choice(["f64", "f64", "f32"])
        n = _log(rng, 8, 1 << 25 if dtype == "f64" else 1024)
        return {"kind": "wave", "dtype": dtype, "n": n,
                "steps": _log(rng, 10, max(11, min(300, int(1e9 / n))))}
    if kind == "audit":
        nx, ny, nz = (_log(rng, 32, 448) for _ in range(3))
        return {"kind": "audit", "dtype": rng.choice(["f32", "f64"]), "nx": nx, "ny": ny, "nz": nz}
    if kind == "host":
        nx, ny, nz = (_log(rng, 32, 224) for _ in range(3))
        return {"kind": "host", "dtype": "f32", "nx": nx, "ny": ny, "nz": nz,
                "steps": rng.randint(1, 8)}
    return {"kind": "train", "records": _log(rng, 100, 4200), "features": rng.randint(20, 48),
            "hidden": 64, "epochs": _log(rng, 50, 400)}


# ------------------------------------------------------------------------------ inputs --------

GAMMA = {"sod": 1.4, "smooth": 1.4, "blast": 1.4, "shear": 5.0 / 3.0}
BCS = {"p": "periodic", "o": "outflow"}
CFL = 0.4


def _shape(case):
    return tuple(case[a] for a in ("nx", "ny", "nz")[:case.get("dim", 3)])


def _primitive(shape, flow, seed):
    """Primitive planes (rho, v, p) in FP64 on the GPU, from the seed alone."""
    rng = np.random.default_rng(seed)
    dim = len(shape)
    axes = [(torch.arange(n, device="cuda", dtype=torch.float64) + 0.5) / n for n in shape]
    X = [c.view([-1 if a == dim - 1 - k else 1 for k in range(dim)]) for a, c in enumerate(axes)]
    V = torch.zeros((dim + 2,) + tuple(reversed(shape)), device="cuda", dtype=torch.float64)
    if flow == "sod":  # the tube's states and position vary a little with the seed
        left = X[0] < rng.uniform(0.45, 0.55)
        V[0] = torch.where(left, rng.uniform(0.95, 1.05), 0.125)
        V[dim + 1] = torch.where(left, rng.uniform(0.95, 1.05), 0.1)
    elif flow == "shear":
        inner = (X[1] - 0.5).abs() < 0.25
        V[0] = torch.where(inner, 2.0, 1.0)
        V[1] = torch.where(inner, 0.5, -0.5)
        V[2] = 0.01 * torch.sin(4.0 * math.pi * X[0] + rng.uniform(0.0, 2.0 * math.pi))
        V[3] = 2.5
    elif flow == "blast":  # a hot sphere of radius eight cells near the centre
        h = 1.0 / max(shape)
        r2 = sum((x - 0.5 - rng.uniform(-2.0, 2.0) * h) ** 2 for x in X)
        V[0] = 1.0
        V[dim + 1] = torch.where(r2 <= (8.0 * h) ** 2, rng.uniform(9.0, 11.0), 1e-3)
    else:  # smooth periodic fields
        def field():
            k = rng.integers(1, 3, size=dim)
            return torch.sin(sum(2.0 * math.pi * float(k[a]) * X[a] for a in range(dim)) +
                             rng.uniform(0.0, 2.0 * math.pi))
        V[0] = 1.25 + 0.75 * field()
        for a in range(dim):
            V[1 + a] = 0.2 * field()
        V[dim + 1] = 1.25 + 0.75 * field()
    return V


def _conserved(V, gamma):
    U = torch.empty_like(V)
    U[0] = V[0]
    U[1:-1] = V[0] * V[1:-1]
    U[-1] = V[-1] / (gamma - 1.0) + 0.5 * V[0] * (V[1:-1] * V[1:-1]).sum(0)
    return U


def _batch_shapes(case):
    """Side lengths drawn log-uniformly, the same ones whenever the case is the same."""
    lo, hi = case["lo"], case["hi"]
    rng = np.random.default_rng([case["grids"], lo, hi])
    s = np.exp(rng.uniform(math.log(lo), math.log(hi), size=(case["grids"], 2)))
    return np.clip(np.rint(s).astype(np.int64), lo, hi)


def _batch_geometry(shapes):
    """For every cell of the packed planes: its grid, x and y (int64 on the GPU)."""
    nx = torch.from_numpy(shapes[:, 0].copy()).cuda()
    ny = torch.from_numpy(shapes[:, 1].copy()).cuda()
    size = nx * ny
    start = torch.cumsum(size, 0) - size
    g = torch.repeat_interleave(torch.arange(len(shapes), device="cuda"), size)
    i = torch.arange(int(size.sum()), device="cuda") - start[g]
    return nx, ny, start, g, i % nx[g], i // nx[g]


def _batch_state(case, seed):
    """Packed conserved planes of smooth periodic data of each grid, FP64."""
    shapes = _batch_shapes(case)
    nx, ny, _, g, x, y = _batch_geometry(shapes)
    rng = np.random.default_rng(seed)
    fx, fy = (x.double() + 0.5) / nx[g], (y.double() + 0.5) / ny[g]
    V = torch.empty((4, len(g)), device="cuda", dtype=torch.float64)
    for k, (mid, amp) in enumerate(((1.25, 0.75), (0.0, 0.2), (0.0, 0.2), (1.25, 0.75))):
        kx, ky = (torch.from_numpy(rng.integers(1, 3, len(shapes)) * 2.0 * math.pi).cuda()
                  for _ in range(2))
        ph = torch.from_numpy(rng.uniform(0.0, 2.0 * math.pi, len(shapes))).cuda()
        V[k] = mid + amp * torch.sin(kx[g] * fx + ky[g] * fy + ph[g])
    return shapes, _conserved(V, 1.4)


def _wave_start(case, seed):
    rng = np.random.default_rng(seed)
    x = torch.arange(case["n"], device="cuda", dtype=torch.float64) * (2.0 * math.pi / case["n"])
    f = torch.sin(x + rng.uniform(0, 6)) + 0.25 * torch.sin(2 * x + rng.uniform(0, 6))
    g = torch.cos(x + rng.uniform(0, 6)) * rng.uniform(0.5, 1.5)
    c = 3.43
    return f, g, c, 2.0 * math.pi, 2.0 * math.pi / case["n"] / c


def _records(case, seed):
    """Feature vectors as the tuner has them (indicator columns, then sizes) and standardised
    log times."""
    rng = np.random.default_rng(seed)
    n, d = case["records"], case["features"]
    X = rng.uniform(0.0, 1.0, (n, d)).astype(np.float32)
    X[:, : d - 6] = (X[:, : d - 6] < 0.2)
    w = rng.normal(0.0, 1.0, d)
    t = X @ w + np.sin(3.0 * X[:, -1]) * X[:, -2] + 0.05 * rng.normal(0.0, 1.0, n)
    return X, ((t - t.mean()) / t.std()).astype(np.float32)


def _state_of(case, seed):
    flow = case.get("flow", "blast")
    V = _primitive(_shape(case), flow, seed)
    return _conserved(V, GAMMA[flow]).to(DTYPES[case["dtype"]])


def _solver(case):
    flow = case.get("flow", "blast")
    dim = case.get("dim", 3)
    return hydro.Solver(_shape(case), GAMMA[flow], bc=[BCS[b] for b in case.get("bc", "p" * dim)],
                        dtype=DTYPES[case["dtype"]], cfl=CFL)


def prepare(case, seed):
    s = dict(case)
    kind = case["kind"]
    if kind == "step":
        s["U0"] = _state_of(case, seed)
        s["U"] = torch.empty_like(s["U0"])
        s["solver"] = _solver(case)
    elif kind == "batch":
        shapes, U = _batch_state(case, seed)
        s["U0"] = U.to(DTYPES[case["dtype"]])
        s["U"] = torch.empty_like(s["U0"])
        s["solver"] = hydro.BatchSolver(shapes, 1.4, dtype=DTYPES[case["dtype"]], cfl=CFL)
    elif kind == "wave":
        f, g, s["c"], s["length"], s["dt"] = _wave_start(case, seed)
        s["f0"], s["g0"] = f.to(DTYPES[case["dtype"]]), g.to(DTYPES[case["dtype"]])
        s["f"], s["g"] = torch.empty_like(s["f0"]), torch.empty_like(s["g0"])
    elif kind == "audit":
        s["U"] = _conserved(_primitive(_shape(case), "smooth", seed), 1.4).to(DTYPES[case["dtype"]])
        s["solver"] = hydro.Solver(_shape(case), 1.4, dtype=DTYPES[case["dtype"]], cfl=CFL)
    elif kind == "host":
        U = _state_of(case, seed)
        s["in"] = torch.empty(U.shape, dtype=U.dtype, pin_memory=True)
        s["in"].copy_(U)
        s["out"] = torch.empty(U.shape, dtype=U.dtype, pin_memory=True)
        s["dev"] = torch.empty_like(U)
        s["solver"] = _solver(case)
    else:
        s["X"], s["t"] = _records(case, seed)
        s["net"] = costmodel.MLP(case["features"], case["hidden"], seed=seed % 1000)
        s["p0"] = s["net"].params.clone()
    return s


def run(s):
    kind = s["kind"]
    real = np.float32 if s.get("dtype") == "f32" else np.float64
    if kind == "step":  # each pass starts from the initial state
        s["U"].copy_(s["U0"])
        t, n = s["solver"].step(s["U"], s["steps"], t_end=s["t_end"])
        return {"U": s["U"], "t": real(t), "steps": n}
    if kind == "batch":
        s["U"].copy_(s["U0"])
        t, n = s["solver"].step(s["U"], s["steps"])
        return {"U": s["U"], "t": np.array(t, dtype=real), "steps": np.array(n)}
    if kind == "wave":
        s["f"].copy_(s["f0"])
        s["g"].copy_(s["g0"])
        e = hydro.wave_run(s["f"], s["g"], s["c"], s["length"], s["dt"], s["steps"])
        return {"f": s["f"], "g": s["g"], "energy": np.array(e, dtype=real)}
    if kind == "audit":
        return {"dt": real(s["solver"].cfl_dt(s["U"])), "totals": np.array(s["solver"].totals(s["U"])),
                "V": hydro.cons_to_prim(s["U"], 1.4)}
    if kind == "host":
        t, n = s["solver"].step_host(s["dev"], s["in"], s["out"], s["steps"])
        return {"out": s["out"], "t": real(t), "steps": n}
    net = s["net"]  # a fresh fit: the initial weights, empty moments
    net.params.copy_(s["p0"])
    net.m.zero_()
    net.v.zero_()
    net.step_count = 0
    loss = net.train(s["X"], s["t"], s["epochs"])
    return {"params": net.params, "m": net.m, "v": net.v, "loss": loss}


# -------------------------------------------------------------------------------- work --------

def _step_flops(dim):
    """Operations of one midpoint-RK step of one cell, every face evaluated once: per stage the
    primitive recovery, per axis the MinBee slopes and face values and one HLLC solve, and the
    update; once per step the CFL signal."""
    nv = dim + 2
    stage = 2 * dim + 5 + dim * (7 * nv + 45 + 5 * dim) + nv * (2 * dim + 1)
    return 2 * stage + 4 * dim + 8


def work(case):
    kind = case["kind"]
    size = 4 if case.get("dtype") == "f32" else 8
    if kind in ("step", "host"):
        dim = case.get("dim", 3)
        cells = math.prod(_shape(case))
        steps = case["steps"]
        if case.get("t_end", 0.0) > 0.0:  # Sod's tube: the fastest wave moves at about 2.2
            steps = min(steps, int(case["t_end"] * 2.2 * case["nx"] / CFL))
        return {"bytes": 2 * (dim + 2) * cells * size, "flops": _step_flops(dim) * cells * steps}
    if kind == "batch":
        # the mean of a log-uniform side, squared
        mean = (case["hi"] - case["lo"]) / math.log(case["hi"] / case["lo"])
        cells = case["grids"] * mean * mean
        return {"bytes": 8 * cells * size, "flops": _step_flops(2) * cells * case["steps"]}
    if kind == "wave":
        return {"bytes": 4 * case["n"] * size, "flops": 14 * case["n"] * case["steps"]}
    if kind == "audit":
        cells = math.prod(_shape(case))
        return {"bytes": 10 * cells * size, "flops": 40 * cells}
    n, d, h = case["records"], case["features"], case["hidden"]
    params = h * d + h + h * h + h + h + 1
    return {"bytes": 4 * (n * (d + 1) + 6 * params),
            "flops": (6 * n * params + 15 * params) * case["epochs"]}


# ------------------------------------------------------------------------------- exact --------

def _flux(L, R, axis, gamma):
    """HLLC flux (Davis speeds) through faces normal to `axis` from their primitive states."""
    u, w = L[1 + axis], R[1 + axis]
    al, ar = (gamma * L[-1] / L[0]).sqrt(), (gamma * R[-1] / R[0]).sqrt()
    SL, SR = torch.minimum(u - al, w - ar), torch.maximum(u + al, w + ar)
    ml, mr = L[0] * (SL - u), R[0] * (SR - w)
    Ss = (R[-1] - L[-1] + u * ml - w * mr) / (ml - mr)
    left = (SL >= 0) | (Ss >= 0)
    star = (SL < 0) & ((Ss >= 0) | (SR > 0))
    S = torch.where(left, SL, SR)
    V = torch.where(left, L, R)
    del L, R, al, ar, SL, SR, ml, mr
    r, p, u = V[0], V[-1], V[1 + axis]
    E = p / (gamma - 1.0) + 0.5 * r * (V[1:-1] * V[1:-1]).sum(0)
    chi = torch.where(star, r * (S - u) / torch.where(star, S - Ss, 1.0), r)
    vs = torch.where(star, Ss, u)
    ps = torch.where(star, p + r * (S - u) * (Ss - u), p)
    es = torch.where(star, ((S - u) * E + ps * Ss - p * u) / torch.where(star, S - Ss, 1.0), E)
    F = torch.empty_like(V)
    m = chi * vs
    F[0] = m
    F[1:-1] = m * V[1:-1]
    F[1 + axis] = m * vs + ps
    F[-1] = vs * (es + ps)
    return F


def _slope(a, b):
    return torch.where(a * b < 0, 0.0, torch.where(a.abs() < b.abs(), a, b))


def _prim(U, gamma):
    V = torch.empty_like(U)
    V[0] = U[0]
    V[1:-1] = U[1:-1] / U[0]
    V[-1] = (gamma - 1.0) * (U[-1] - 0.5 * U[0] * (V[1:-1] * V[1:-1]).sum(0))
    return V


def _rates(U, gamma, bc, dr):
    """-sum_a dF_a/dr_a of a whole grid, ghost cells by wrapping or copying the end cells."""
    V = _prim(U, gamma)
    out = torch.zeros_like(U)
    for a in range(len(dr)):
        d = U.dim() - 1 - a
        n = U.shape[d]
        i = torch.arange(-2, n + 2, device=U.device)
        P = V.index_select(d, i % n if bc[a] == "p" else i.clamp(0, n - 1))
        D = P.narrow(d, 1, n + 3) - P.narrow(d, 0, n + 3)
        s = _slope(D.narrow(d, 0, n + 2), D.narrow(d, 1, n + 2))
        del D
        C = P.narrow(d, 1, n + 2)
        L = (C + 0.5 * s).narrow(d, 0, n + 1)
        R = (C - 0.5 * s).narrow(d, 1, n + 1)
        del P, C, s
        F = _flux(L, R, a, gamma)
        del L, R
        out += (F.narrow(d, 0, n) - F.narrow(d, 1, n)) / dr[a]
        del F
    return out


def _exact_steps(U, gamma, bc, shape, steps, t_end):
    U = U.double().clone()
    dr = [1.0 / n for n in shape]
    t, done = 0.0, 0
    while done < steps and not (t_end > 0.0 and t >= t_end):
        V = _prim(U, gamma)
        cs = (gamma * V[-1] / V[0]).sqrt()
        dt = CFL / float(sum((V[1 + a].abs() + cs) / dr[a] for a in range(len(dr))).max())
        del V, cs
        last = t_end > 0.0 and dt >= t_end - t
        dt = t_end - t if last else dt
        U1 = U + 0.5 * dt * _rates(U, gamma, bc, dr)
        U += dt * _rates(U1, gamma, bc, dr)
        t, done = (t_end if last else t + dt), done + 1
    return U, t, done


def _exact_batch(case, seed):
    shapes, U = _batch_state(case, seed)
    U = U.to(DTYPES[case["dtype"]]).double()
    nx, ny, start, g, x, y = _batch_geometry(shapes)
    dr = [1.0 / nx[g].double(), 1.0 / ny[g].double()]
    near = []  # cells at -2 ... 2 along each axis, periodic
    for a, (c, n, other) in enumerate(((x, nx, y), (y, ny, x))):
        row = []
        for k in (-2, -1, 1, 2):
            j = (c + k) % n[g]
            row.append(start[g] + (other * nx[g] + j if a == 0 else j * nx[g] + other))
        near.append(row)

    def rates(W):
        V = _prim(W, 1.4)
        out = torch.zeros_like(W)
        for a in range(2):
            q = [V[:, i] for i in near[a]]
            q.insert(2, V)
            d = [q[k + 1] - q[k] for k in range(4)]
            s = [_slope(d[k], d[k + 1]) for k in range(3)]
            out += (_flux(q[1] + 0.5 * s[0], q[2] - 0.5 * s[1], a, 1.4) -
                    _flux(q[2] + 0.5 * s[1], q[3] - 0.5 * s[2], a, 1.4)) / dr[a]
        return out

    t = torch.zeros(len(shapes), device="cuda", dtype=torch.float64)
    for _ in range(case["steps"]):
        V = _prim(U, 1.4)
        cs = (1.4 * V[-1] / V[0]).sqrt()
        sig = (V[1].abs() + cs) / dr[0] + (V[2].abs() + cs) / dr[1]
        most = torch.zeros_like(t).scatter_reduce(0, g, sig, "amax")
        dt = CFL / most
        U1 = U + 0.5 * dt[g] * rates(U)
        U = U + dt[g] * rates(U1)
        t = t + dt
    return {"U": U, "t": t, "steps": None}


def _exact_train(case, seed):
    X, y = (torch.from_numpy(a).double().cuda() for a in _records(case, seed))
    d, h, n = case["features"], case["hidden"], case["records"]
    flat = costmodel.MLP(d, h, seed=seed % 1000).params.double()  # the initial weights
    size = [h * d, h, h * h, h, h, 1]
    m, v, loss = torch.zeros_like(flat), torch.zeros_like(flat), []
    for k in range(1, case["epochs"] + 1):
        W1, b1, W2, b2, W3, b3 = torch.split(flat, size)
        W1, W2 = W1.view(h, d), W2.view(h, h)
        h1 = torch.tanh(X @ W1.T + b1)
        h2 = torch.tanh(h1 @ W2.T + b2)
        e = h2 @ W3 + b3 - y
        loss.append((e * e).mean())
        dy = 2.0 * e / n
        z2 = dy[:, None] * W3 * (1.0 - h2 * h2)
        z1 = (z2 @ W2) * (1.0 - h1 * h1)
        grad = torch.cat([(z1.T @ X).reshape(-1), z1.sum(0), (z2.T @ h1).reshape(-1), z2.sum(0),
                          dy @ h2, dy.sum().reshape(1)])
        m = 0.9 * m + 0.1 * grad
        v = 0.999 * v + 0.001 * grad * grad
        flat = flat - 3e-3 * (m / (1.0 - 0.9 ** k)) / ((v / (1.0 - 0.999 ** k)).sqrt() + 1e-8)
    return {"params": flat, "m": m, "v": v, "loss": torch.stack(loss)}


def exact(case, seed):
    kind = case["kind"]
    if kind == "step":
        U, t, _ = _exact_steps(_state_of(case, seed), GAMMA[case["flow"]], case["bc"],
                               _shape(case), case["steps"], case["t_end"])
        return {"U": U, "t": np.float64(t), "steps": None}
    if kind == "host":
        U, t, _ = _exact_steps(_state_of(case, seed), 1.4, "ppp", _shape(case), case["steps"], 0.0)
        return {"out": U, "t": np.float64(t), "steps": None}
    if kind == "batch":
        return _exact_batch(case, seed)
    if kind == "wave":
        f, g, c, length, dt = _wave_start(case, seed)
        f, g = (a.to(DTYPES[case["dtype"]]).double() for a in (f, g))
        dx = length / case["n"]
        energy = []
        for _ in range(case["steps"]):
            f = f + dt * g
            up, down = f.roll(-1), f.roll(1)
            h = g + c * c * dt / (dx * dx) * (up + down - 2.0 * f)
            energy.append((c * c * ((up - down) / (2.0 * dx)).square() +
                           (0.5 * (g + h)).square()).sum() * 0.5 * dx)
            g = h
        return {"f": f, "g": g, "energy": torch.stack(energy)}
    if kind == "audit":
        U = _conserved(_primitive(_shape(case), "smooth", seed), 1.4).to(DTYPES[case["dtype"]]).double()
        V = _prim(U, 1.4)
        shape = _shape(case)
        cs = (1.4 * V[-1] / V[0]).sqrt()
        dt = CFL / sum((V[1 + a].abs() + cs) * shape[a] for a in range(3)).max()
        vol = 1.0 / math.prod(shape)
        return {"dt": dt, "totals": torch.stack([U[k].sum() * vol for k in range(5)]), "V": V}
    return _exact_train(case, seed)
