"""What the framework's speed is measured on: the work of the immersed-boundary LES a user has it do.

Every case goes through the public binding (paper_2002_06206_gb300/ibmles.py).  The kinds of work:

  step      one whole fractional step (les_step): a run is nothing but thousands of these
  momentum  the momentum half of a step: eddy viscosity, predictor (Crank-Nicolson with its implicit
            solve, or Adams-Bashforth 2) and the distributed forcing, on a body standing in the stream
  project   the projection around the pressure solve: face velocities, right-hand side, correction
  solve     the pressure Poisson solve alone, which dominates a step
  classify  per-geometry set-up: ray-cast classification of a triangle soup and its link records
  train     one training step of the learned pressure guess (forward, backward, Adam)

The physics, boundary types, solver settings and soups are those of the repository's workloads, tests
and benchmark: CFL 0.2, 10 % QUICK, multigrid-preconditioned CG in FP32 inside FP64 refinement with
residual checks every 8 iterations and 1e-5 per refinement, or everything in FP64.

The exact values below are plain torch in 64 bits, written from the scheme's definition for a body whose
cut links are known in closed form (an axis-aligned box), for a pressure that is known beforehand, and
for soups small enough to test every triangle against every grid line.
"""
import functools
import math

import numpy as np
import torch

import workloads as W
from paper_2002_06206_gb300 import ibmles as L

BC = {"channel": W.configs.CHANNEL, "ground": W.configs.GROUND, "span": (1, 2, 0, 0, 3, 3)}
DEV = "cuda"
F64 = torch.float64
CFL, QUICK = 0.2, 0.1


# ---- the cases -----------------------------------------------------------------------------------

def listed():
    return [
        # the small validation run: a clean sphere at Re = 100 in FP64, Adams-Bashforth, to 1e-10; the
        # smallest whole call, where launches and latency count
        {"name": "step_sphere_fp64", "kind": "step", "body": "sphere", "nx": 64, "ny": 32, "nz": 32, "fp64": True,
         "integrator": "ab2", "bc": "channel", "re": 100.0, "tol": 1e-10},
        # the benchmark's headline: a vehicle-like dirty assembly of 2 M triangles in ground effect, 201 M cells
        {"name": "step_vehicle", "kind": "step", "body": "vehicle", "nx": 1024, "ny": 512, "nz": 384, "fp64": False,
         "integrator": "cn", "bc": "ground", "re": 1.5e5, "tol": 1e-6},
        # Crank-Nicolson momentum on the bluff-body grid: the implicit solve of the production integrator
        {"name": "momentum_cn", "kind": "momentum", "nx": 512, "ny": 256, "nz": 256, "fp64": False,
         "integrator": "cn", "bc": "ground", "dx": 1.0},
        # explicit predictor on an odd grid: no row starts on a vector boundary
        {"name": "momentum_ab2_odd", "kind": "momentum", "nx": 251, "ny": 127, "nz": 93, "fp64": False,
         "integrator": "ab2", "bc": "channel", "dx": 1.0},
        # the momentum half in FP64, as validation runs take it
        {"name": "momentum_cn_fp64", "kind": "momentum", "nx": 128, "ny": 64, "nz": 64, "fp64": True,
         "integrator": "cn", "bc": "channel", "dx": 1.0},
        # face velocities, right-hand side and correction on the bluff-body grid
        {"name": "project", "kind": "project", "nx": 512, "ny": 256, "nz": 256, "fp64": False, "bc": "ground",
         "dx": 1.0},
        # the pressure solve of the bluff-body and dirty-sphere workloads (mixed precision, multigrid)
        {"name": "solve_cube", "kind": "solve", "body": "box", "nx": 512, "ny": 256, "nz": 256, "fp64": False,
         "bc": "ground", "solver": "mg"},
        {"name": "solve_dirty_sphere", "kind": "solve", "body": "dirty", "nx": 256, "ny": 128, "nz": 128,
         "fp64": False, "bc": "channel", "solver": "mg"},
        # the same on an odd grid
        {"name": "solve_odd", "kind": "solve", "body": "dirty", "nx": 131, "ny": 61, "nz": 47, "fp64": False,
         "bc": "channel", "solver": "mg"},
        # classification and set-up of the vehicle assembly (every new geometry pays it)
        {"name": "classify_vehicle", "kind": "classify", "body": "vehicle", "nx": 1024, "ny": 512, "nz": 384},
        # ... and of the 1280-triangle sphere, the smallest geometry
        {"name": "classify_sphere", "kind": "classify", "body": "sphere", "nx": 64, "ny": 32, "nz": 32},
        # one training step of the learned pressure guess on a 128^3 patch
        {"name": "train", "kind": "train", "nx": 128, "ny": 128, "nz": 128, "lr": 1e-3},
    ]


def _dims(rng, lo, hi):
    """A grid of about lo .. hi cells (log-uniform), longer along x as a channel is, odd sizes among them."""
    cells = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    ay, az = rng.uniform(0.35, 0.8), rng.uniform(0.3, 0.7)
    nx = (cells / (ay * az)) ** (1.0 / 3.0)
    n = [max(24, int(nx)), max(16, int(ay * nx)), max(16, int(az * nx))]
    kind = rng.randrange(3)
    if kind == 0:                                   # the multiples most users take
        n = [max(32, 16 * round(v / 16)) for v in n]
    elif kind == 1:                                 # ragged
        n = [v | 1 for v in n]
    return dict(zip(("nx", "ny", "nz"), n))


def draw(rng):
    kind = rng.choice(["step", "momentum", "momentum", "project", "solve", "solve", "classify", "train"])
    fp64 = rng.random() < 0.3
    if kind == "step":
        c = _dims(rng, 4e4, 1e6 if fp64 else 1.6e7)
        return {"kind": kind, "body": rng.choice(["sphere", "dirty", "vehicle"]), **c, "fp64": fp64,
                "integrator": "cn", "bc": rng.choice(["channel", "ground"]),
                "re": round(math.exp(rng.uniform(math.log(100.0), math.log(2e4))), 1), "tol": 1e-10 if fp64 else 1e-6}
    if kind == "momentum":
        return {"kind": kind, **_dims(rng, 4e4, 2e6 if fp64 else 3e7), "fp64": fp64,
                "integrator": rng.choice(["cn", "ab2"]), "bc": rng.choice(["channel", "ground", "span"]),
                "dx": rng.choice([1.0, 0.5])}
    if kind == "project":
        return {"kind": kind, **_dims(rng, 1e5, 3e7), "fp64": fp64, "bc": rng.choice(["channel", "ground", "span"]),
                "dx": rng.choice([1.0, 0.5])}
    if kind == "solve":
        c = _dims(rng, 4e4, 2e6 if fp64 else 3e7)
        return {"kind": kind, "body": rng.choice(["box", "sphere", "dirty"]), **c, "fp64": fp64,
                "bc": rng.choice(["channel", "ground"]),
                "solver": rng.choice(["mg", "mg", "mg", "cg" if c["nx"] * c["ny"] * c["nz"] < 3e6 else "mg"])}
    if kind == "classify":
        return {"kind": kind, "body": rng.choice(["sphere", "dirty", "vehicle"]), **_dims(rng, 4e4, 1e8)}
    return {"kind": kind, **_dims(rng, 3e4, 4e6), "lr": rng.choice([1e-3, 3e-4])}


# ---- inputs --------------------------------------------------------------------------------------

def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


def _randn(shape, g, dtype=F64):
    return torch.randn(shape, generator=g, device=DEV, dtype=dtype)


@functools.lru_cache(maxsize=4)
def _base_soup(body, nx, ny, nz):
    """A workload's soup, sized to the grid (float64 [ntri, 3, 3], grid units); the seed only moves it."""
    if body == "vehicle":
        s = min(nx / 1024.0, ny / 512.0, nz / 384.0)
        lo, hi = (0.19 * nx, 0.27 * ny, 0.05 * nz), (0.81 * nx, 0.73 * ny, 0.05 * nz + 0.42 * nz)
        t = W.vehicle_assembly(seed=4, target_tris=max(3000, int(2_000_000 * s * s)), envelope_lo=(192.0, 136.0, 16.0),
                               envelope_hi=(832.0, 376.0, 176.0)).astype(np.float64)
        a, b = np.array([192.0, 136.0, 16.0]), np.array([832.0, 376.0, 176.0])
        if (nx, ny, nz) != (1024, 512, 384):
            t = (t - a) / (b - a) * (np.array(hi) - np.array(lo)) + np.array(lo)
        return t
    r = min(nx, ny, nz) / 8.0
    cen = (0.25 * nx, 0.5 * ny, 0.5 * nz)
    if body == "dirty":
        return W.dirty_sphere(seed=2, radius=r, center=cen, subdiv=5 if r > 10.0 else 4).astype(np.float64)
    return W.icosphere(3 if r < 8.0 else 5, r, cen, dtype=np.float64)


def _soup(case, seed):
    """The case's soup on the device, shifted by a seeded fraction of a cell; for the classification alone
    by whole cells (on a 2^-13 lattice, so that every shift is exact), which keeps the number of cut faces."""
    if case["body"] == "box":
        return torch.from_numpy(W.axis_box(*_box(case, seed), 8)).to(DEV)
    t = _base_soup(case["body"], case["nx"], case["ny"], case["nz"])
    rng = np.random.default_rng(seed)
    if case["kind"] == "classify":
        m = np.maximum(1, np.array([case["nx"], case["ny"], case["nz"]]) // 32)
        return torch.from_numpy((np.round(t * 8192.0) / 8192.0 + rng.integers(-m, m + 1)).astype(np.float32)).to(DEV)
    return torch.from_numpy((t + rng.uniform(-0.5, 0.5, 3)).astype(np.float32)).to(DEV)


def _box(case, seed):
    """Corners of a box body off the cell centres, on the floor for the ground boundary types."""
    n = np.array([case["nx"], case["ny"], case["nz"]])
    f = np.random.default_rng(seed).uniform(0.1, 0.4, 6)
    lo = np.floor(n * np.array([0.22, 0.44, 0.38])) + f[:3]
    hi = np.floor(n * np.array([0.29, 0.56, 0.62])) + 0.5 + f[3:]
    if case["bc"] == "ground":
        lo[2], hi[2] = 0.0, math.floor(0.125 * n[2]) + 0.5 + f[5]
    return lo.astype(np.float32).astype(np.float64), hi.astype(np.float32).astype(np.float64)


def _modes(case, seed, n, kmax, slope, shift=0.0):
    """n random plane-wave products on the cell centres, amplitudes falling as k^-slope, moved by `shift`
    cells along x: [nz, ny, nx] in FP64, RMS about 1."""
    rng = np.random.default_rng(seed)
    dims = (case["nz"], case["ny"], case["nx"])
    out = torch.zeros(dims, device=DEV, dtype=F64)
    norm = 0.0
    for _ in range(n):
        k = np.exp(rng.uniform(0.0, math.log(kmax), 3))
        a = np.linalg.norm(k) ** -slope
        ph = rng.uniform(0.0, 2.0 * math.pi, 3)
        f = []
        for q, m in enumerate(dims):
            x = torch.arange(m, device=DEV, dtype=F64) + 0.5 - (shift if q == 2 else 0.0)
            f.append(torch.cos(math.pi * min(k[q], m / 4.0) / m * x + ph[q]))
        out += a * f[0][:, None, None] * f[1][None, :, None] * f[2][None, None, :]
        norm += a * a / 8.0
    return out / math.sqrt(norm)


def _velocity(case, seed, shift, inside):
    """The stream (1, 0, 0) with eddies of 10 % and small noise, at rest in the body: [3, nz, ny, nx]."""
    g = _gen(seed)
    u = torch.stack([0.1 * _modes(case, 7 * seed + c, 6, 24.0, 0.8, shift) for c in range(3)])
    u += 1e-3 * _randn(u.shape, g)
    u[0] += 1.0
    return torch.where(inside, torch.zeros((), device=DEV, dtype=F64), u)


def _axes(case):
    z, y, x = (torch.arange(case[k], device=DEV, dtype=F64) + 0.5 for k in ("nz", "ny", "nx"))
    return x[None, None, :], y[None, :, None], z[:, None, None]


def _inside_box(case, seed):
    lo, hi = _box(case, seed)
    r = None
    for a, x in enumerate(_axes(case)):
        m = (x > lo[a]) & (x < hi[a])
        r = m if r is None else r & m
    return r


def _pressure(case, seed):
    """A pressure with a range of scales that is zero inside the body and its sealed pockets, where the
    equation fixes it up to a constant only: [nz, ny, nx] in FP64."""
    p = 0.2 * _modes(case, seed, 12, 32.0, 1.5)
    if case.get("body", "box") == "box":
        inside = _inside_box(case, seed)
    else:                                           # a ball a little larger than the (jittered) sphere
        r = min(case["nx"], case["ny"], case["nz"]) / 8.0 * 1.01 + 1.0
        d = np.random.default_rng(seed).uniform(-0.5, 0.5, 3)
        c = (0.25 * case["nx"] + d[0], 0.5 * case["ny"] + d[1], 0.5 * case["nz"] + d[2])
        inside = sum((x - c[a]) ** 2 for a, x in enumerate(_axes(case))) < r * r
    return torch.where(inside, torch.zeros((), device=DEV, dtype=F64), p)


def _grid(case):
    return L.make_grid(case["nx"], case["ny"], case["nz"], case.get("dx", 1.0))


def _nu(case):
    return case.get("dx", 1.0) * min(case["nx"], case["ny"], case["nz"]) / 4.0 / case.get("re", 1e4)


def _solver(case, geo, tol=1e-6):
    precond = L.NO_PRECOND if case.get("solver") == "cg" else L.MULTIGRID
    cn = case.get("integrator") == "cn"
    return L.Solver(_grid(case), _nu(case), CFL * case.get("dx", 1.0), BC[case["bc"]],
                    precision=L.FP64 if case["fp64"] else L.FP32_REFINE64, tol=tol, check_every=8, inner_tol=1e-5,
                    geometry=geo, precond=precond, quick=QUICK if cn or case["kind"] == "momentum" else 0.0,
                    integrator=L.CRANK_NICOLSON if cn else L.ADAMS_BASHFORTH)


def prepare(case, seed):
    kind = case["kind"]
    s = {"kind": kind, "case": case}
    n = (case["nz"], case["ny"], case["nx"])
    N = n[0] * n[1] * n[2]
    if kind == "classify":
        s["grid"], s["tri"] = _grid(case), _soup(case, seed)
        return s
    if kind == "train":
        s["grid"] = _grid(case)
        b, p, dp, ddp = _snapshot(case, seed)
        s["b"], s["p"], s["pp"] = b, p, p - dp
        s["flags"] = (_inside_ball(case, seed) * 3).to(torch.uint8).reshape(-1)
        s["target"] = ddp.to(torch.float32)
        s["net"] = L.Net(_net_params(seed))
        return s
    if kind == "step":
        geo = L.Geometry(_grid(case), _soup(case, seed), deadend_on=int(case["body"] == "vehicle"))
        solver = _solver(case, geo, case["tol"])
        g = _gen(seed)
        u0 = torch.empty((3, N), device=DEV, dtype=solver.dtype)
        for c in range(3):
            u0[c] = 1e-3 * _randn((N,), g, solver.dtype) + (1.0 if c == 0 else 0.0)
        s["solver"], s["st"] = solver, solver.fields(u0)
        return s
    body = dict(case, body=case.get("body", "box"))
    geo = L.Geometry(_grid(case), _soup(body, seed))
    tol = 1e-11 if kind == "solve" else 1e-6
    solver = s["solver"] = _solver(case, geo, tol)
    dt = solver.dtype
    if kind == "solve":
        s["tol"] = tol
        s["b"] = torch.empty(N, device=DEV, dtype=F64)
        solver.apply(_pressure(body, seed).reshape(-1).contiguous(), s["b"])
        s["p"] = torch.zeros(N, device=DEV, dtype=F64)
        return s
    if kind == "momentum":
        # two instants of one flow, a time step apart, taken in turn: the implicit solve of a step starts
        # from the last step's increment, which belongs to a slightly different field
        s["u"], s["U"], s["turn"] = [], [], 0
        for q in range(2):
            u = _velocity(case, seed, CFL * q, _inside_box(case, seed)).to(dt).reshape(-1).contiguous()
            U = torch.empty(solver.NF, device=DEV, dtype=dt)
            solver.init_faces(u, U)
            s["u"].append(u)
            s["U"].append(U)
        s["nut"] = torch.empty(N, device=DEV, dtype=dt)
        s["Hprev"] = (0.01 * _randn((3 * N,), _gen(seed + 1))).to(dt)
        s["H"] = torch.empty(3 * N, device=DEV, dtype=dt)
        s["ustar"] = torch.empty(3 * N, device=DEV, dtype=dt)
        return s
    s["ustar"] = _velocity(case, seed, 0.0, _inside_box(case, seed)).to(dt).reshape(-1).contiguous()
    s["p"] = _pressure(body, seed).reshape(-1).contiguous()
    s["Ustar"] = torch.empty(solver.NF, device=DEV, dtype=dt)
    s["b"] = torch.empty(N, device=DEV, dtype=F64)
    s["u"] = torch.empty(3 * N, device=DEV, dtype=dt)
    s["U"] = torch.empty(solver.NF, device=DEV, dtype=dt)
    return s


def run(s):
    kind = s["kind"]
    if kind == "classify":
        geo = L.Geometry(s["grid"], s["tri"])
        out = {"flags": geo.flags, "face_id": geo.face_id, "t_lo": geo.t_lo, "t_hi": geo.t_hi}
        geo.close()
        return out
    if kind == "train":
        net = s["net"]
        loss = net.train_step(s["grid"], s["b"], s["p"], s["pp"], s["target"], s["case"]["lr"], s["flags"])
        # the loss is a sum of FP32 terms, as the network's outputs are
        return {"loss": np.float32(loss), "grads": net.grads(), "params": net.params()}
    solver = s["solver"]
    if kind == "step":
        st = s["st"]
        solver.step(st)
        out = {"u": st["u"], "U": st["U"]}
        if s["case"]["fp64"]:
            out["p"] = st["p"]
        # in the mixed-precision mode p is left out: inside the soup's sealed pockets the equation fixes it up
        # to a constant only, which two runs on the same inputs do not share; u and U hold its gradient
        return out
    if kind == "solve":
        s["p"].zero_()
        solver.solve(s["b"], s["p"], s["tol"])
        return {"p": s["p"]}
    if kind == "momentum":
        q = s["turn"]
        s["turn"] = 1 - q
        u, U = s["u"][q], s["U"][q]
        solver.csm(u, s["nut"])
        if s["case"]["integrator"] == "cn":
            solver.predict_cn(u, U, s["nut"], s["H"], s["ustar"])
        else:
            solver.predict(u, U, s["nut"], s["Hprev"], s["H"], s["ustar"], False)
        solver.forcing(s["ustar"])
        return {"nut": s["nut"], "H": s["H"], "ustar": s["ustar"]}
    solver.faces(s["ustar"], s["Ustar"])
    solver.rhs(s["Ustar"], s["b"])
    solver.correct(s["ustar"], s["Ustar"], s["p"], s["u"], s["U"])
    return {"Ustar": s["Ustar"], "b": s["b"], "u": s["u"], "U": s["U"]}


def work(case):
    """Bytes: every input of the pass read once and every output written once.  Operations: the stencil
    arithmetic of one application where the path is one (a solve's count depends on its method)."""
    N = case["nx"] * case["ny"] * case["nz"]
    w = 8 if case.get("fp64") else 4
    kind = case["kind"]
    if kind == "step":                # u, U, p, flags in; u, U, p, H out (H in too with Adams-Bashforth)
        return {"bytes": N * (15 * w + 16 + 1 + (3 * w if case["integrator"] == "ab2" else 0)), "flops": 500 * N}
    if kind == "momentum":            # u, U, flags (Hprev) in; nut, H, u* out
        return {"bytes": N * (13 * w + 1 + (3 * w if case["integrator"] == "ab2" else 0)), "flops": 330 * N}
    if kind == "project":             # u*, p, flags in; U*, b, u, U out
        return {"bytes": N * (3 * w + 8 + 1 + 3 * w + 8 + 6 * w), "flops": 25 * N}
    if kind == "solve":               # b, flags in; p out
        return {"bytes": 17 * N, "flops": 15 * N}
    if kind == "classify":            # the soup in; flags and the region bits and record index of each cell out
        return {"bytes": 36 * len(_base_soup(case["body"], case["nx"], case["ny"], case["nz"])) + 5 * N, "flops": 0}
    # b, p, p_prev, flags, target in; the convolutions forward, back and by weight
    return {"bytes": N * 29, "flops": 2 * N * 27 * (8 * 8 * 3 + 8 * 8 * 3 + 8 * 3)}


# ---- the learned guess's snapshot -------------------------------------------------------------------

def _snapshot(case, seed):
    b = 0.05 * _modes(case, seed + 1, 10, 32.0, 0.5) + 0.01 * _randn((case["nz"], case["ny"], case["nx"]), _gen(seed))
    p = 0.3 * _modes(case, seed + 2, 10, 16.0, 1.5)
    dp = 0.01 * _modes(case, seed + 3, 10, 24.0, 1.0) + 1e-3 * _randn(b.shape, _gen(seed + 1))
    ddp = 0.5 * _modes(case, seed + 4, 10, 24.0, 1.0)
    return [v.reshape(-1).contiguous() for v in (b, p, dp, ddp)]


def _inside_ball(case, seed):
    r = min(case["nx"], case["ny"], case["nz"]) / 8.0
    d = np.random.default_rng(seed).uniform(-0.5, 0.5, 3)
    c = (0.25 * case["nx"] + d[0], 0.5 * case["ny"] + d[1], 0.5 * case["nz"] + d[2])
    rr = sum((x - c[a]) ** 2 for a, x in enumerate(_axes(case))).sqrt()
    return (rr - r).abs() < 0.6                    # the shell of cells with a cut link


def _net_params(seed):
    rng = np.random.default_rng(seed)
    return np.concatenate([rng.standard_normal(m) * 0.1 for m in (1728, 1728, 216)] +
                          [rng.standard_normal(m) * 0.05 for m in (8, 8, 1)]).astype(np.float32)


# ---- exact values -----------------------------------------------------------------------------------

def exact(case, seed):
    kind = case["kind"]
    if kind == "solve":
        body = dict(case, body=case.get("body", "box"))
        return {"p": _pressure(body, seed).reshape(-1)}
    if kind == "momentum":
        return _exact_momentum(case, seed)
    if kind == "project":
        return _exact_project(case, seed)
    if kind == "train":
        return _exact_train(case, seed)
    if kind == "classify":
        return _exact_classify(case, seed)
    return None                                     # a whole step: many coupled solves


class _Links:
    """The links of the grid around a box body: which are cut and how far the wall is, in closed form;
    values across a link by the ghost rule of the scheme.  Arrays are [nz, ny, nx]; axis a of the grid is
    array dimension 2 - a."""

    def __init__(self, case, seed):
        lo, hi = _box(case, seed)
        self.n = n = (case["nx"], case["ny"], case["nz"])
        self.bc = BC[case["bc"]]
        ax = _axes(case)
        self.cut, self.d, self.out = {}, {}, {}
        shape = (n[2], n[1], n[0])
        for a in range(3):
            b, c = (a + 1) % 3, (a + 2) % 3
            line = (ax[b] > lo[b]) & (ax[b] < hi[b]) & (ax[c] > lo[c]) & (ax[c] < hi[c])
            for s in (-1, 1):
                end = ax[a] + s
                inside = (end > 0) & (end < n[a])
                cut = torch.zeros(shape, device=DEV, dtype=torch.bool)
                d = torch.zeros(shape, device=DEV, dtype=F64)
                for w in (lo[a], hi[a]):
                    dist = s * (w - ax[a])
                    hit = line & inside & (dist >= 0) & (dist < 1) & torch.ones(shape, device=DEV, dtype=torch.bool)
                    cut |= hit
                    d = torch.where(hit, dist.expand(shape), d)
                self.cut[a, s], self.d[a, s] = cut, d
                self.out[a, s] = (~inside).expand(shape) & (self.bc[2 * a] != 0)
        self.coef = {}
        for a in range(3):
            for s in (-1, 1):
                d, ok = self.d[a, s], ~self.out[a, -s] & ~self.cut[a, -s]
                back = ax[a] - s
                ok = ok & ((back > 0) & (back < n[a])).expand(shape)     # a link across a periodic seam is no partner
                near = (d < 0.5) & ok
                one = torch.ones_like(d)
                cp = torch.where(d >= 0.5, (d - 1) / torch.where(d > 0, d, one), torch.where(near, -2 * d, -one))
                self.coef[a, s] = (cp, torch.where(near, 2 * d - 1, torch.zeros_like(d)))

    @staticmethod
    def shift(f, a, s):
        return torch.roll(f, -s, 2 - a)

    def across(self, f, comp, a, s, hom=False):
        v = self.shift(f, a, s)
        bc = self.bc[2 * a + (s > 0)]
        if bc != 0:
            uin = 1.0 if comp == 0 and not hom else 0.0
            g = 2 * uin - f if bc == 1 else f if bc == 2 else (-f if comp == a else f) if bc == 3 else -f
            v = torch.where(self.out[a, s], g, v)
        cp, co = self.coef[a, s]
        return torch.where(self.cut[a, s], cp * f + co * self.shift(f, a, -s), v)

    def face(self, U, a, s):
        """The face value of each cell's link (a, s) from the face array of axis a."""
        m = self.n[a]
        return U[a].narrow(2 - a, 1 if s > 0 else 0, m)

    def split(self, U):
        out, o = [], 0
        for a in range(3):
            m = [self.n[2], self.n[1], self.n[0]]
            m[2 - a] += 1
            c = m[0] * m[1] * m[2]
            out.append(U[o:o + c].reshape(m))
            o += c
        return out


def _faces64(K, u):
    """Face velocities of a cell field: mean on open faces, 0 on cut ones and walls, the boundary value on
    domain faces, the outflow shifted to zero net flux."""
    out = []
    for a in range(3):
        m = K.n[a]
        dim = 2 - a
        up = 0.5 * (u[a] + K.shift(u[a], a, 1))
        up = torch.where(K.cut[a, 1], torch.zeros_like(up), up)
        first, last = u[a].narrow(dim, 0, 1), u[a].narrow(dim, m - 1, 1)
        seam = 0.5 * (last + first)
        ends = []
        for s, v in ((-1, first), (1, last)):
            bc = K.bc[2 * a + (s > 0)]
            ends.append(seam if bc == 0 else torch.full_like(v, 1.0 if a == 0 else 0.0) if bc == 1 else
                        v if bc == 2 else torch.zeros_like(v))
        out.append(torch.cat([ends[0], up.narrow(dim, 0, m - 1), ends[1]], dim))
    net, cnt = 0.0, 0
    for a in range(3):
        for s in (-1, 1):
            v = out[a].narrow(2 - a, 0 if s < 0 else K.n[a], 1)
            if K.bc[2 * a + (s > 0)] in (1, 2):
                net = net + s * v.sum()
            cnt += v.numel() if K.bc[2 * a + (s > 0)] == 2 else 0
    for a in range(3):
        for s in (-1, 1):
            if K.bc[2 * a + (s > 0)] == 2:
                out[a].narrow(2 - a, 0 if s < 0 else K.n[a], 1).sub_(s * net / cnt)
    return out


def _flux64(K, u, U, nut, nu, dx, gam, hom):
    """Momentum operator per cell: flux-form advection (central with a share of QUICK), diffusion with
    nu + nu_t, the transposed part of the sub-grid stress."""
    G = [[(K.across(u[c], c, a, 1, hom) - K.across(u[c], c, a, -1, hom)) / (2 * dx) for c in range(3)] for a in range(3)]
    h = [torch.zeros_like(nut) for _ in range(3)]
    for a in range(3):
        for s in (-1, 1):
            Uf = K.face(U, a, s)
            inner = ~K.cut[a, s] & ~K.out[a, s]
            nutf = torch.where(inner, 0.5 * (nut + K.shift(nut, a, s)), nut)
            for c in range(3):
                v = K.across(u[c], c, a, s, hom)
                D1 = (v - u[c]) / dx
                Tt = D1
                if c != a:
                    Tt = s * torch.where(inner, 0.5 * (G[c][a] + K.shift(G[c][a], a, s)), G[c][a])
                adv = 0.5 * (u[c] + v)
                if gam:
                    lo, hi = (u[c], v) if s > 0 else (v, u[c])
                    flo, fhi = K.across(u[c], c, a, -1, hom), K.across(u[c], c, a, 1, hom)
                    if s > 0:
                        fhi = K.shift(fhi, a, 1)
                    else:
                        flo = K.shift(flo, a, -1)
                    q = torch.where(Uf >= 0, 6 * lo + 3 * hi - flo, 6 * hi + 3 * lo - fhi) / 8
                    adv = torch.where(inner, (1 - gam) * adv + gam * q, adv)
                h[c] += -s * Uf * adv + (nu + nutf) * D1 + nutf * Tt
    return torch.stack(h) / dx


def _csm64(K, u, dx):
    G = [[(K.across(u[c], c, a, 1) - K.across(u[c], c, a, -1)) / (2 * dx) for c in range(3)] for a in range(3)]
    SS = WW = 0.0
    for a in range(3):
        for b in range(3):
            SS = SS + (0.5 * (G[a][b] + G[b][a])) ** 2
            WW = WW + (0.5 * (G[a][b] - G[b][a])) ** 2
    E = 0.5 * (WW + SS)
    Fc = torch.where(E > 0, 0.5 * (WW - SS) / torch.where(E > 0, E, torch.ones_like(E)), torch.zeros_like(E)).abs()
    return Fc ** 1.5 / 20.0 * dx * dx * SS.sqrt()


def _forcing64(K, us):
    add, wsum = torch.zeros_like(us), torch.zeros_like(us[0])
    for (a, s), cut in K.cut.items():
        d = K.d[a, s]
        w = torch.where(cut, (1 - d) / (1 + d), torch.zeros_like(d))
        wsum = wsum + w
        for c in range(3):
            add[c] -= w * ((1 - d) * us[c] + d * K.shift(us[c], a, s))
    return us + add / wsum.clamp(min=1.0)


def _exact_momentum(case, seed):
    K = _Links(case, seed)
    work_dt = F64 if case["fp64"] else torch.float32
    u = _velocity(case, seed, 0.0, _inside_box(case, seed)).to(work_dt).to(F64)
    # the faces of the state are its inputs: in the working precision, from the cell field's rule
    U = [f.to(work_dt).to(F64) for f in _faces64(K, u)]
    dx, dt, nu = case["dx"], CFL * case["dx"], _nu(case)
    nut = _csm64(K, u, dx)
    H = _flux64(K, u, U, nut, nu, dx, QUICK, False)
    if case["integrator"] == "cn":
        # delta = dt L(u) + dt/2 L0(delta): contracting at this CFL number
        delta = dt * H
        for _ in range(60):
            new = dt * H + 0.5 * dt * _flux64(K, delta, U, nut, nu, dx, QUICK, True)
            step = float((new - delta).norm() / new.norm())
            delta = new
            if step < (1e-13 if case["fp64"] else 1e-10):
                break
        us = u + delta
    else:
        Hp = (0.01 * _randn((3 * nut.numel(),), _gen(seed + 1))).to(work_dt).to(F64).reshape(u.shape)
        us = u + dt * (1.5 * H - 0.5 * Hp)
    return {"nut": nut.reshape(-1), "H": H.reshape(-1), "ustar": _forcing64(K, us).reshape(-1)}


def _exact_project(case, seed):
    K = _Links(case, seed)
    work_dt = F64 if case["fp64"] else torch.float32
    us = _velocity(case, seed, 0.0, _inside_box(case, seed)).to(work_dt).to(F64)
    p = _pressure(dict(case, body="box"), seed)
    dx = case["dx"]
    dt = CFL * dx
    Us = _faces64(K, us)
    b, u, U = 0.0, [], []
    for a in range(3):
        dim, m = 2 - a, K.n[a]
        b = b + (K.face(Us, a, 1) - K.face(Us, a, -1)) / (dx * dt)
        v = {}
        for s in (-1, 1):
            bc = K.bc[2 * a + (s > 0)]
            x = K.shift(p, a, s)
            if bc != 0:
                x = torch.where(K.out[a, s], -p if bc == 2 else p, x)
            v[s] = torch.where(K.cut[a, s], p, x)
        u.append(us[a] - dt / (2 * dx) * (v[1] - v[-1]))
        hi, lo = v[1] - p, p - v[-1]              # zero on cut faces and walls: those keep their U*
        hi, lo = (torch.where(K.out[a, s] & (K.bc[2 * a + (s > 0)] == 1), torch.zeros_like(p), g)
                  for s, g in ((1, hi), (-1, lo)))
        grad = torch.cat([lo.narrow(dim, 0, 1), hi], dim)
        U.append(Us[a] - dt / dx * grad)
    flat = lambda f: torch.cat([x.reshape(-1) for x in f])  # noqa: E731
    return {"Ustar": flat(Us), "b": b.reshape(-1), "u": torch.stack(u).reshape(-1), "U": flat(U)}


def _exact_train(case, seed):
    n = (case["nz"], case["ny"], case["nx"])
    b, p, dp, ddp = _snapshot(case, seed)
    dp = p - (p - dp)
    dx = case.get("dx", 1.0)
    scale = dp.square().mean().sqrt()
    flags = _inside_ball(case, seed).reshape(-1).to(F64)
    x = torch.zeros((1, 8) + n, device=DEV, dtype=F64)
    for c, v in enumerate((b * dx * dx / scale, dp / scale, flags)):
        x[0, c] = v.reshape(n)
    th = torch.from_numpy(_net_params(seed)).to(DEV, F64).requires_grad_(True)
    w = [th[:1728].view(8, 27, 8), th[1728:3456].view(8, 27, 8), th[3456:3672].view(1, 27, 8)]
    bias = [th[3672:3680], th[3680:3688], th[3688:3689]]
    y = x
    for q in range(3):
        k = w[q].permute(0, 2, 1).reshape(-1, 8, 3, 3, 3)
        y = torch.nn.functional.conv3d(y, k, bias[q], padding=1)
        y = y.relu() if q < 2 else y
    loss = (y.reshape(-1) - ddp.to(torch.float32).to(F64)).square().mean()
    g, = torch.autograd.grad(loss, th)
    new = th.detach() - case["lr"] * g / (g.abs() + 1e-8)       # Adam's first step: m / c1 = g, v / c2 = g^2
    return {"loss": loss.detach(), "grads": g, "params": new}


def _exact_classify(case, seed):
    n = (case["nx"], case["ny"], case["nz"])
    N = n[0] * n[1] * n[2]
    tri = _soup(case, seed).to(F64)
    if len(tri) * sum(n[a] * n[(a + 1) % 3] for a in range(3)) > 4e9:
        return None                                 # every triangle against every line would take too long
    st = (1, n[0], n[0] * n[1])
    ids, ts = [], []
    for a in range(3):
        b, c = (a + 1) % 3, (a + 2) % 3
        qb = torch.arange(n[b], device=DEV, dtype=F64)[None, :, None] + 0.5
        qc = torch.arange(n[c], device=DEV, dtype=F64)[None, None, :] + 0.5
        chunk = max(1, int(1.5e7 / (n[b] * n[c])))
        for t0 in range(0, len(tri), chunk):
            V = tri[t0:t0 + chunk]
            A, B, C = (V[:, q, :, None, None] for q in range(3))
            orient = lambda P, Q: (Q[:, b] - P[:, b]) * (qc - P[:, c]) - (Q[:, c] - P[:, c]) * (qb - P[:, b])  # noqa: E731
            w = [orient(B, C), orient(C, A), orient(A, B)]
            Wt = (w[0] + w[1]) + w[2]
            thr = -1e-9 * Wt.abs()
            sg = torch.sign(Wt)
            hit = (Wt != 0) & (sg * w[0] >= thr) & (sg * w[1] >= thr) & (sg * w[2] >= thr)
            q, jb, jc = hit.nonzero(as_tuple=True)
            if not len(q):
                continue
            num = (w[0][q, jb, jc] * A[q, a, 0, 0] + w[1][q, jb, jc] * B[q, a, 0, 0]) + w[2][q, jb, jc] * C[q, a, 0, 0]
            xm = num / Wt[q, jb, jc] - 0.5
            f = xm.floor()
            ok = (f >= 0) & (f <= n[a] - 2)
            cell = f.to(torch.int64) * st[a] + jb * st[b] + jc * st[c]
            ids.append((a * N + cell)[ok])
            ts.append((xm - f)[ok])
    face, inv = torch.unique(torch.cat(ids), return_inverse=True)
    t = torch.cat(ts)
    lo = torch.full((len(face),), 2.0, device=DEV, dtype=F64).scatter_reduce(0, inv, t, "amin")
    hi = torch.full((len(face),), -1.0, device=DEV, dtype=F64).scatter_reduce(0, inv, t, "amax")
    return {"flags": None, "face_id": None, "t_lo": lo, "t_hi": hi}
