"""The work a user has this framework do, as cases that can be timed and compared.

Kinds of case:

* ``solve``: one blocking ``mcgrav_solve`` (host stations in, host results out)
  over the sphere, the prism, the paper's cube in a ball, or a voxel model
  with tabulated boundary data, in the mixed or the plain FP64 walk;
* ``walk`` : the device-level path (``DeviceSolve``: walk, reduce, finalize),
  which hands back every path's own values;
* ``field``: the exact field of a density model (``mcg_field``);
* ``model``: the set-up of a heterogeneous model (``voxel_model``: the random
  density and its six boundary tables);
* ``serve``: a batch of requests through a running server.

The geometries are those of ``paper_1709_07469_gb300.workloads``; the seed
moves the stations a little, seeds the walks and makes the density.
"""
import math

import numpy as np
import torch

from paper_1709_07469_gb300 import mcgrav as M
from paper_1709_07469_gb300 import workloads as W
from paper_1709_07469_gb300.device import DeviceSolve, voxel_model

DEV = "cuda"


def listed():
    return [
        # a first check of an installation, or one evaluation inside a script's loop: latency
        {"name": "sphere_check", "kind": "solve", "model": "sphere", "precision": "mixed", "stations": 8,
         "paths": 256, "step": math.sqrt(1e-3), "bridge": 0, "crn": 1},
        # a quick look at a survey line over the ore body, at the benchmark's 1 m step
        {"name": "prism_quick", "kind": "solve", "model": "prism", "precision": "mixed", "stations": 30,
         "paths": 256, "step": 1.0, "bridge": 0, "crn": 1},
        # one batch of the benchmark's ore-body survey
        {"name": "prism_survey", "kind": "solve", "model": "prism", "precision": "mixed", "stations": 30,
         "paths": 8192, "step": 1.0, "bridge": 0, "crn": 1},
        # coarse steps with the exit-time correction, a ragged batch, every path's own values
        {"name": "prism_walk_bridge", "kind": "walk", "model": "prism", "precision": "mixed", "stations": 7,
         "paths": 1001, "step": 5.0, "bridge": 1, "crn": 1},
        # the heterogeneous model under a 16 x 16 station grid
        {"name": "voxel_survey", "kind": "solve", "model": "voxel", "precision": "mixed", "stations": 256,
         "paths": 512, "step": 10.0, "bridge": 0, "crn": 1, "nx": 128, "ny": 128, "nz": 64, "table": 64},
        # the same model under a dense ground and airborne survey, few paths at each of many stations
        {"name": "large_survey", "kind": "solve", "model": "survey", "precision": "mixed", "stations": 20000,
         "paths": 32, "step": 10.0, "bridge": 0, "crn": 1, "nx": 128, "ny": 128, "nz": 64, "table": 64},
        # the paper's own experiment: a cube in a large ball with zero data
        {"name": "cube_ball", "kind": "solve", "model": "ball", "precision": "mixed", "stations": 31,
         "paths": 512, "step": 20.0, "bridge": 0, "crn": 1},
        # the plain double-precision walk, the check on the mixed one: its smallest problem ...
        {"name": "sphere_fp64", "kind": "solve", "model": "sphere", "precision": "fp64", "stations": 8,
         "paths": 2000, "step": math.sqrt(1e-3), "bridge": 0, "crn": 1},
        # ... and the ore body
        {"name": "prism_fp64", "kind": "solve", "model": "prism", "precision": "fp64", "stations": 30,
         "paths": 256, "step": 10.0, "bridge": 0, "crn": 1},
        # the exact field of the voxel model at the survey's stations, to compare estimates with
        {"name": "field_voxel", "kind": "field", "model": "voxel", "points": 256, "nx": 128, "ny": 128, "nz": 64},
        # a new random subsurface and its boundary tables: once per model
        {"name": "model_setup", "kind": "model", "nx": 128, "ny": 128, "nz": 64, "table": 128},
        # an inversion code's burst of requests on two resident models
        {"name": "serve_burst", "kind": "serve", "requests": 12, "max_stations": 16, "target": 1e-2,
         "nx": 64, "ny": 64, "nz": 32, "table": 33},
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _int(rng, lo, hi):
    return max(lo, min(hi, int(round(_log(rng, lo, hi)))))


# steps of a drawn case at most, below those of the largest listed ones
MAX_STEPS = {"mixed": 1.0e10, "fp64": 5e6}


def draw(rng):
    kind = rng.choice(["solve", "solve", "solve", "solve", "walk", "field", "model", "serve"])
    if kind == "field":
        if rng.random() < 0.25:
            return {"kind": "field", "model": "prism", "points": _int(rng, 100, 1000000)}
        nx, ny, nz = rng.randint(16, 128), rng.randint(16, 128), rng.randint(8, 64)
        return {"kind": "field", "model": "voxel", "points": _int(rng, 1, 256), "nx": nx, "ny": ny, "nz": nz}
    if kind == "model":
        n = rng.randint(24, 128)
        return {"kind": "model", "nx": n, "ny": rng.randint(24, 128), "nz": max(8, n // 2),
                "table": _int(rng, 9, 128)}
    if kind == "serve":
        n = rng.choice([16, 32, 48, 64])
        return {"kind": "serve", "requests": _int(rng, 1, 12), "max_stations": _int(rng, 1, 16),
                "target": rng.choice([1e-2, 2e-2]), "nx": n, "ny": n, "nz": n // 2, "table": rng.randint(9, 65)}
    # the plain walk's plain form is the common one; the others are the mixed walk's
    precision = "fp64" if rng.random() < 0.25 else "mixed"
    model = rng.choice(["sphere", "prism"] if precision == "fp64" else ["sphere", "prism", "ball", "voxel"])
    case = {"kind": kind, "model": model, "precision": precision, "stations": _int(rng, 1, 300),
            "paths": _int(rng, 32, 20000)}
    lo, hi = {"sphere": (0.015, 0.06), "prism": (1.0, 20.0), "ball": (20.0, 100.0), "voxel": (10.0, 40.0)}[model]
    if precision == "fp64" and model == "prism":
        lo = 10.0
    case["step"] = _log(rng, lo, hi)
    case["bridge"] = int(model in ("sphere", "prism") and rng.random() < 0.2)
    case["crn"] = int(rng.random() < 0.85)
    if model == "voxel":
        n = rng.randint(16, 128)
        case.update(nx=n, ny=rng.randint(16, 128), nz=max(8, n // 2), table=rng.randint(9, 65))
    per_path = _mean_steps(case)
    case["paths"] = max(1, min(case["paths"], int(MAX_STEPS[precision] / per_path / case["stations"])))
    case["stations"] = max(1, min(case["stations"], int(MAX_STEPS[precision] / per_path / case["paths"])))
    return case


# --- problems --------------------------------------------------------------------

def _voxel_shape(case):
    return (case["nx"], case["ny"], case["nz"])


def _workload(case):
    """The repository's workload of a case, with its own station layout."""
    m, step = case["model"], case.get("step", 10.0)
    if m == "sphere":
        w = W.sphere_line(dt=step * step)
    elif m == "prism":
        w = W.prism_ore_body(step=step)
    elif m == "ball":
        w = W.paper_cube_ball(step=step)
    else:
        t = case.get("table", 9)
        make = W.large_survey if m == "survey" else W.voxel_survey
        w = make(step=step, shape=_voxel_shape(case), table_n=(t, t))
    return w.with_(bridge=case.get("bridge", 0), crn=case.get("crn", 1), paths=case.get("paths", 1))


def _stations(case, w, seed, n):
    """`n` of the workload's stations (in turn, more than once if need be),
    each moved by up to a hundredth of the layout's spacing."""
    rng = np.random.default_rng([seed, 17])
    k = np.arange(n) * max(1, w.n_stations // n) % w.n_stations
    scale = 5e-4 if w.name == "sphere_line" else 0.5
    return w.stations[k] + rng.uniform(-scale, scale, (n, 3))


def _grid(seed, shape, amp=300.0):
    """A smooth lognormal density on the voxel grid, [nz, ny, nx] float32."""
    nx, ny, nz = shape
    g = torch.Generator(device=DEV).manual_seed(seed)
    z = torch.randn((1, 1, nz, ny, nx), generator=g, device=DEV, dtype=torch.float64)
    for _ in range(3):
        z = torch.nn.functional.avg_pool3d(z, 5, 1, 2, count_include_pad=False)
    z = z[0, 0]
    return (amp * torch.expm1((z - z.mean()) / z.std(correction=0))).float().contiguous()


def _voxel_problem(w, grid):
    """Grid and boundary tables of a voxel workload, on the device."""
    nu, nv = w.table_n
    faces = torch.empty((6, nv, nu), dtype=torch.float32, device=DEV)
    M.mcg_boundary_tables(M.problem(w.with_(g_kind="zero"), grid=grid), nu, nv, 4.0, faces)
    return faces


class _Server:
    """A server and its resident models, given back with the state."""

    def __init__(self, case, seed):
        case = dict(case, model="voxel")
        self.w = w = _workload(case)
        self.models = []
        for k in range(2):
            grid = _grid(seed + 1000 * k, _voxel_shape(case))
            p = M.problem(w, grid=grid, faces=_voxel_problem(w, grid))
            torch.cuda.synchronize()
            self.models.append(M.mcg_model_create(p, w.dt, w.h))
        self.server = M.mcg_server_create(M.server_config(M.options(w)))
        rng = np.random.default_rng([seed, 5])
        self.requests = []
        for r in range(case["requests"]):
            S = 1 + (7 * r + 3) % case["max_stations"]
            st = w.stations[rng.choice(w.n_stations, size=S, replace=False)]
            self.requests.append((self.models[r % 2], st, case["target"] * (1.0 if r % 3 else 0.5), seed + r))

    def __del__(self):
        if getattr(self, "server", None):
            M.mcg_server_destroy(self.server)
        for m in getattr(self, "models", ()):
            M.mcg_model_destroy(m)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "serve":
        return {"kind": kind, "server": _Server(case, seed)}
    if kind == "model":
        t = case["table"]
        w = W.voxel_survey(shape=_voxel_shape(case), table_n=(t, t), grid_seed=seed)
        return {"kind": kind, "w": w}
    w = _workload(case)
    if kind == "field":
        n = case["points"]
        g = torch.Generator(device=DEV).manual_seed(seed)
        lo, hi = torch.tensor(w.lo, device=DEV).double(), torch.tensor(w.hi, device=DEV).double()
        x = lo + (hi - lo) * torch.rand((n, 3), generator=g, device=DEV, dtype=torch.float64)
        grid = None
        if case["model"] == "voxel":
            x[:, 2] = 0.01 * x[:, 2].abs()     # stations at and above the surface
            w = w.with_(g_kind="zero")
            grid = _grid(seed, _voxel_shape(case))
        return {"kind": kind, "prob": M.problem(w, grid=grid), "x": x, "n": n, "w": w, "grid": grid}
    w = w.with_(seed=seed)
    st = _stations(case, w, seed, case["stations"])
    grid = faces = None
    if w.rho_kind == "voxel":
        grid = _grid(seed, _voxel_shape(case))
        faces = _voxel_problem(w, grid)
    precision = M.MCG_FP64 if case["precision"] == "fp64" else M.MCG_MIXED
    if kind == "walk":
        ds = DeviceSolve(w, stations=st, batch=case["paths"], precision=precision, grid=grid, faces=faces)
        return {"kind": kind, "ds": ds}
    return {"kind": kind, "prob": M.problem(w, grid=grid, faces=faces), "st": st, "w": w,
            "opts": M.options(w, precision=precision), "paths": case["paths"]}


def run(state):
    kind = state["kind"]
    if kind == "solve":
        w = state["w"]
        r = M.mcgrav_solve(state["prob"], state["st"], state["paths"], w.dt, w.seed, state["opts"])
        return _solved(w.crn, vars(r))
    if kind == "walk":
        ds = state["ds"]
        ds.reset()
        ds.walk(0)
        ds.reduce()
        ds.finalize()
        crn = ds.w.crn
        return {"pp_u": ds.pp_u, "pp_d": ds.pp_d if crn else None, "pp_steps": ds.pp_steps,
                "res": ds.res[:4] if crn else ds.res[0:3:2], "counts": ds.res[4:].view(torch.int64),
                "status": ds.status}
    if kind == "field":
        phi = torch.empty(state["n"], dtype=torch.float64, device=DEV)
        gz = torch.empty_like(phi)
        M.mcg_field(state["prob"], state["x"], state["n"], phi, gz)
        return {"phi": phi, "gz": gz}
    if kind == "model":
        grid, faces = voxel_model(state["w"])
        return {"grid": grid, "faces": faces}
    sv = state["server"]
    handles = [(M.mcg_submit(sv.server, m, st, target, seed), len(st)) for m, st, target, seed in sv.requests]
    out = []
    for h, S in handles:
        rc, r = M.mcg_wait(h, S)
        M.mcg_request_free(h)
        if rc != M.MCG_OK:
            raise M.McgError(rc, "request failed")
        out.append(np.stack([r[k] for k in ("u", "gz", "se_u", "se_gz")]))
        out.append(np.stack([r["n_paths"], r["path_steps"]]))
    return out


def _solved(crn, r):
    keys = ["u", "se_u", "n_paths", "path_steps"] + (["gz", "se_gz"] if crn else [])
    return {k: r[k] for k in keys}


# --- what a case cannot do without ------------------------------------------------

def _mean_steps(case):
    """Mean number of steps of a walk from the middle of the workload's
    stations: the mean exit time of a Brownian motion over dt."""
    w = _workload(dict(case, bridge=0))
    x = w.stations.mean(axis=0)
    if w.domain == "ball":
        return (w.ball_radius ** 2 - float(np.sum((x - np.array(w.ball_center)) ** 2))) / 3.0 / w.dt
    L = np.array(w.hi) - np.array(w.lo)
    t = np.concatenate([[0.0], np.geomspace(1e-6, 20.0, 4000) * L.min() ** 2])
    n = np.arange(1, 400, 2)[:, None]
    surv = np.ones_like(t)
    for k in range(3):     # survival of each coordinate: its sine series
        a = 4.0 / (n * np.pi) * np.sin(n * np.pi * (x[k] - w.lo[k]) / L[k])
        surv = surv * np.sum(a * np.exp(-0.5 * (n * np.pi / L[k]) ** 2 * t), axis=0).clip(0.0, 1.0)
    return float(np.trapezoid(surv, t)) / w.dt


def work(case):
    kind = case["kind"]
    cells = case.get("nx", 0) * case.get("ny", 0) * case.get("nz", 0)
    if kind == "field":
        # prism: eight corners; voxel: one corner function per grid node and point
        nodes = 8 if case["model"] == "prism" else (case["nx"] + 1) * (case["ny"] + 1) * (case["nz"] + 1)
        return {"bytes": 40.0 * case["points"] + 4.0 * cells, "flops": 45.0 * nodes * case["points"]}
    if kind == "model":
        # every node of the tables sees every cell (distance, reciprocal root, multiply-add)
        nodes = 6 * case["table"] ** 2
        return {"bytes": 4.0 * (cells + nodes), "flops": 8.0 * nodes * cells + 200.0 * cells}
    per_step = 74.0        # operations of one step of the three copies: generator, normals, move, tests, sums
    if kind == "serve":
        steps = _mean_steps(dict(case, model="voxel"))
        S = 0.5 * (case["max_stations"] + 1) * case["requests"]
        return {"bytes": 72.0 * S + 2 * 4.0 * (cells + 6 * case["table"] ** 2),
                "flops": per_step * steps * S * 8192.0}
    n = float(case["stations"] * case["paths"])
    out = 24.0 * n if kind == "walk" else 0.0
    tables = 4.0 * 6 * case["table"] ** 2 if cells else 0.0
    return {"bytes": out + 72.0 * case["stations"] + 4.0 * cells + tables,
            "flops": (per_step if case["crn"] else 62.0) * n * _mean_steps(case)}


# --- the same in 64 bits, by plain torch -------------------------------------------

def _philox(ctr, key):
    """Philox4x32-10 (Salmon et al. 2011) on int64 tensors holding 32-bit words."""
    m = 0xFFFFFFFF

    def wide(a, x):      # high and low word of the 64-bit product, by 16-bit halves of a
        lo, hi = (a & 0xFFFF) * x, (a >> 16) * x
        mid = hi + (lo >> 16)
        return mid >> 16, ((mid & 0xFFFF) << 16) | (lo & 0xFFFF)

    c0, c1, c2, c3 = ctr
    k0, k1 = key
    for _ in range(10):
        h0, l0 = wide(0xD2511F53, c0)
        h1, l1 = wide(0xCD9E8D57, c2)
        c0, c1, c2, c3 = h1 ^ c1 ^ k0, l1, h0 ^ c3 ^ k1, l0
        k0, k1 = (k0 + 0x9E3779B9) & m, (k1 + 0xBB67AE85) & m
    return c0, c1, c2, c3


def _gauss(w1, w2, bits):
    """Box-Muller pair of two words, from their leading `bits` bits."""
    u1, u2 = (((w >> (32 - bits)).double() + 0.5) * 2.0 ** -bits for w in (w1, w2))
    r, a = torch.sqrt(-2.0 * torch.log(u1)), 2.0 * math.pi * u2
    return r * torch.cos(a), r * torch.sin(a)


def _corner(x, y, z):
    """Corner function of the prism potential and its z derivative."""
    r = torch.sqrt(x * x + y * y + z * z)

    def ln(t, p, q):     # log(t + r) without cancellation
        return torch.where(t >= 0, torch.log(torch.where(t >= 0, t + r, torch.ones_like(r))),
                           torch.log(p * p + q * q) - torch.log(r - t))

    def term(c, f):      # a term with a vanishing factor is 0
        return torch.where(c != 0, c * f, torch.zeros_like(f))

    lx, ly, lz = ln(x, y, z), ln(y, z, x), ln(z, x, y)
    az = torch.atan(x * y / (z * r))
    F = term(x * y, lz) + term(y * z, lx) + term(z * x, ly)
    F = F - term(0.5 * x * x, torch.atan(y * z / (x * r))) - term(0.5 * y * y, torch.atan(z * x / (y * r)))
    return F - term(0.5 * z * z, az), term(x, ly) + term(y, lx) - term(z, az)


def _prism(lo, hi, x):
    """Sums of the corner function and its derivative over a prism's corners, seen from points x [..., 3]."""
    f, d = 0.0, 0.0
    for c in range(8):
        i, j, k = c & 1, (c >> 1) & 1, (c >> 2) & 1
        F, D = _corner((hi, lo)[1 - i][0] - x[..., 0], (hi, lo)[1 - j][1] - x[..., 1], (hi, lo)[1 - k][2] - x[..., 2])
        s = -1.0 if (3 - i - j - k) & 1 else 1.0
        f, d = f + s * F, d + s * D
    return f, d


def _node_sum(grid, w, x):
    """Potential and vertical gravity of a voxel grid at points x, by grid nodes."""
    g = torch.nn.functional.pad(grid.double(), (1, 1, 1, 1, 1, 1))
    for k in range(3):
        g = g.narrow(k, 0, g.shape[k] - 1) - g.narrow(k, 1, g.shape[k] - 1)
    nz, ny, nx = g.shape
    ax = [w.grid_origin[k] + w.grid_spacing[k] * torch.arange(n, device=DEV).double()
          for k, n in enumerate((nx, ny, nz))]
    phi, gz = torch.empty(len(x), device=DEV).double(), torch.empty(len(x), device=DEV).double()
    for i in range(len(x)):
        F, D = _corner((ax[0] - x[i, 0])[None, None, :].expand(nz, ny, nx), (ax[1] - x[i, 1])[None, :, None],
                       (ax[2] - x[i, 2])[:, None, None])
        phi[i], gz[i] = -w.G * (g * F).sum(), w.G * (g * D).sum()
    return phi, gz


def _density(w, X):
    if w.rho_kind == "sphere":
        c = torch.tensor(w.center, device=DEV).double()
        inside = ((X - c) ** 2).sum(-1) < w.radius ** 2
    else:
        lo, hi = torch.tensor(w.plo, device=DEV).double(), torch.tensor(w.phi, device=DEV).double()
        inside = ((X >= lo) & (X < hi)).all(-1)
    return w.rho0 * inside.double()


def _boundary(w, X):
    if w.rho_kind == "sphere":       # the boundary lies outside the sphere
        c = torch.tensor(w.center, device=DEV).double()
        return -w.G * (4.0 / 3.0 * math.pi * w.radius ** 3 * w.rho0) / (X - c).norm(dim=-1)
    return -w.G * w.rho0 * _prism(w.plo, w.phi, X)[0]


def _walks64(w, st, paths, bits):
    """Every walk of S stations x paths in 64 bits: u and its copies [n, C], steps [n]."""
    S, C = len(st), 3 if w.crn else 1
    n, sd = S * paths, w.sigma * math.sqrt(w.dt)
    off = torch.tensor([0.0, w.h, -w.h][:C], device=DEV).double()
    lo, hi = torch.tensor(w.lo, device=DEV).double(), torch.tensor(w.hi, device=DEV).double()
    key = (w.seed & 0xFFFFFFFF, (w.seed >> 32) & 0xFFFFFFFF)
    sid = torch.arange(S, device=DEV).repeat_interleave(paths)
    pid = torch.arange(paths, device=DEV).repeat(S)
    W0 = torch.from_numpy(st).to(DEV)[sid]
    shift = torch.zeros((C, 3), device=DEV).double()
    shift[:, 2] = off
    rp = _density(w, W0[:, None] + shift)
    integral = torch.zeros((n, C), device=DEV).double()
    u, steps = torch.zeros((n, C), device=DEV).double(), torch.zeros(n, dtype=torch.int64, device=DEV)
    live = torch.ones((n, C), dtype=torch.bool, device=DEV)
    at, b0 = torch.arange(n, device=DEV), 0
    while len(at):
        B = max(1, min(64, 500000 // len(at)))
        j = (3 * b0 + torch.arange(3 * B, device=DEV))[None, :].expand(len(at), 3 * B)
        p, s = pid[at][:, None].expand_as(j), sid[at][:, None].expand_as(j)
        x0, x1, x2, x3 = _philox((j, p, s, torch.zeros_like(j)), key)
        z = torch.stack(_gauss(x0, x1, bits) + _gauss(x2, x3, bits), -1).reshape(len(at), 4 * B, 3)
        path = torch.cat([W0[at][:, None], W0[at][:, None] + torch.cumsum(sd * z, 1)], 1)
        X = path[:, :, None] + shift                      # [m, T + 1, C, 3]
        out = ~((X[:, 1:] > lo) & (X[:, 1:] < hi)).all(-1)
        T = 4 * B
        first = torch.where(out.any(1), out.int().argmax(1), T)       # [m, C] step that leaves, or T
        rho = torch.cat([rp[at][:, None], _density(w, X[:, 1:])], 1)  # [m, T + 1, C]
        k = torch.arange(T, device=DEV)[None, :, None]
        part = (0.5 * (rho[:, :-1] + rho[:, 1:]) * (k < first[:, None])).sum(1) * w.dt
        alive = live[at]
        integral[at] += torch.where(alive, part, 0.0)
        steps[at] += torch.where(alive, torch.clamp(first + 1, max=T), 0).sum(1)
        gone = alive & (first < T)
        if gone.any():
            r, c = gone.nonzero(as_tuple=True)
            f = first[r, c]
            a, b, ra = X[r, f, c], X[r, f + 1, c], rho[r, f, c]
            wall = torch.where(b <= lo, lo, hi)
            th = torch.where((b <= lo) | (b >= hi), (wall - a) / (b - a), torch.inf)
            t, axis = th.min(-1, keepdim=True)
            xs = (a + t.clamp(0.0, 1.0) * (b - a)).scatter(1, axis, wall.gather(1, axis))
            rest = 0.5 * (ra + _density(w, xs)) * t[:, 0].clamp(0.0, 1.0) * w.dt
            u[at[r], c] = _boundary(w, xs) - 2.0 * math.pi * w.G * (integral[at[r], c] + rest)
        live[at] = alive & (first == T)
        rp[at], W0[at] = rho[:, -1], path[:, -1]
        at = at[live[at].any(1)]
        b0 += B
    return u, steps


def exact(case, seed):
    kind = case["kind"]
    if kind == "serve" or (kind in ("solve", "walk") and (case["bridge"] or case["model"] in ("ball", "voxel", "survey"))):
        return None      # long walks whose steps are single precision: no path of theirs has a 64-bit value
    if kind == "field":
        st = prepare(case, seed)
        if case["model"] == "voxel":
            phi, gz = _node_sum(st["grid"], st["w"], st["x"])
        else:
            f, d = _prism(st["w"].plo, st["w"].phi, st["x"])
            phi, gz = -st["w"].G * st["w"].rho0 * f, st["w"].G * st["w"].rho0 * d
        return {"phi": phi, "gz": gz}
    if kind == "model":
        return _exact_model(case, seed)
    # the mixed walk decides its exits in single precision: only means of short walks have a 64-bit value
    mixed = case["precision"] == "mixed"
    total = case["stations"] * case["paths"] * _mean_steps(case)
    if total > (2e7 if mixed and case["model"] == "sphere" else 0 if mixed else 2e8):
        return None
    w = _workload(case).with_(seed=seed)
    st = _stations(case, w, seed, case["stations"])
    u, steps = _walks64(w, st, case["paths"], 23 if mixed else 32)
    S, N = case["stations"], case["paths"]
    d = (u[:, 1] - u[:, 2]) / (2.0 * w.h) if w.crn else torch.full_like(u[:, 0], math.nan)
    u0, dd = u[:, 0].reshape(S, N), d.reshape(S, N)
    mean = {"u": u0.mean(1), "gz": dd.mean(1), "se_u": torch.sqrt(u0.var(1) / N), "se_gz": torch.sqrt(dd.var(1) / N)}
    counts = torch.stack([torch.full((S,), N, device=DEV), steps.reshape(S, N).sum(1)])
    if mixed:
        mean["gz"] = mean["se_gz"] = None
    if kind == "walk":
        if mixed:        # whole per-path values, which single precision moves one by one
            return None
        res = torch.stack([mean[k] for k in (("u", "gz", "se_u", "se_gz") if w.crn else ("u", "se_u"))])
        return {"pp_u": u[:, 0], "pp_d": d if w.crn else None, "pp_steps": steps, "res": res, "counts": counts,
                "status": torch.zeros(2, dtype=torch.int32)}
    return _solved(w.crn, dict(mean, n_paths=counts[0], path_steps=counts[1]))


def _exact_model(case, seed):
    nx, ny, nz = _voxel_shape(case)
    t = case["table"]
    w = W.voxel_survey(shape=(nx, ny, nz), table_n=(t, t), grid_seed=seed)
    n = nx * ny * nz
    q = torch.arange((n + 3) // 4, device=DEV)
    zero = torch.zeros_like(q)
    x0, x1, x2, x3 = _philox((q, zero, zero, zero + 1), (seed & 0xFFFFFFFF, (seed >> 32) & 0xFFFFFFFF))
    a = torch.stack(_gauss(x0, x1, 32) + _gauss(x2, x3, 32), -1).reshape(-1)[:n].reshape(nz, ny, nx)
    R = math.ceil(3.0 * w.grid_sigma_vox)
    taps = np.exp(-np.arange(-R, R + 1) ** 2 / (2.0 * w.grid_sigma_vox ** 2))
    taps = taps / taps.sum()
    for axis in (2, 1, 0):
        b = torch.zeros_like(a)
        L = a.shape[axis]
        for m, c in zip(range(-R, R + 1), taps):
            if abs(m) < L:
                b.narrow(axis, max(0, -m), L - abs(m)).add_(a.narrow(axis, max(0, m), L - abs(m)), alpha=float(c))
        a = b
    grid = w.grid_amp * torch.expm1((a - a.mean()) / a.std(correction=0))
    faces = None
    if 6 * t * t * (nx + 1) * (ny + 1) * (nz + 1) < 5e8:
        s = torch.linspace(0.0, 1.0, t, device=DEV).double()
        lo, hi = torch.tensor(w.lo, device=DEV).double(), torch.tensor(w.hi, device=DEV).double()
        x = torch.empty((6, t, t, 3), device=DEV).double()
        for f in range(6):
            k = f >> 1
            ua, va = (1, 2) if k == 0 else (0, 2) if k == 1 else (0, 1)
            x[f, :, :, k] = (hi if f & 1 else lo)[k]
            x[f, :, :, ua] = (lo[ua] + (hi[ua] - lo[ua]) * s)[None, :]
            x[f, :, :, va] = (lo[va] + (hi[va] - lo[va]) * s)[:, None]
        faces = _node_sum(grid.float(), w, x.reshape(-1, 3))[0].reshape(6, t, t)
    return {"grid": grid, "faces": faces}
