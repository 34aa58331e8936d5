"""Workloads of this library as its users run them, for timing and for comparing outputs.

A case is a dict of plain values: the kind of program, the model, the storage form, the
grid (nx, ny, nz), the number of lattice steps and the relaxation frequency, and what a
kind needs beyond that.  The kinds are the programs that the entry points serve:

  host      a small run from numpy arrays through the Lattice class, fields read back
  run       device fields -> lbm_init -> lbm_step -> the stored state (lbm_get_raw), and for
            the FP32 and FP64 forms the macroscopic fields (lbm_moments)
  tube      the same with fixed end states (lbm_set_fixed_ends), the shock-tube set-up
  restart   populations of another program -> lbm_set_populations -> lbm_step ->
            lbm_get_populations
  gradient  a differentiable rollout (autograd.rollout) under a squared loss, and its
            backward pass to the initial fields

Every grid holds a planar Riemann problem (two states on either side of a diaphragm) with
smooth seeded perturbations of density, velocity and temperature and white density noise.
exact() is a plain torch restatement in 64 bits of the paper's update (fourth-order Hermite
equilibrium on D2Q33 / D3Q95, BGK relaxation, pull streaming on a periodic box); it uses
nothing of the package.
"""
from __future__ import annotations

import itertools
import math

import numpy as np
import torch

DEVICE = "cuda"
BYTES = {"fp64": 8, "fp32": 4, "fp16": 2, "bf16": 2}
RAW = {"fp64": torch.float64, "fp32": torch.float32, "fp16": torch.float16,
       "bf16": torch.bfloat16}
DIM = {"D2Q33": 2, "D3Q95": 3}
NQ = {"D2Q33": 33, "D3Q95": 95}


# ------------------------------------------------------------------ the cases
def _case(kind, model, storage, nx, ny, nz, steps, omega, **more):
    return dict(kind=kind, model=model, storage=storage, nx=nx, ny=ny, nz=nz, steps=steps,
                omega=omega, **more)


def listed():
    def named(name, *a, **k):
        return dict(_case(*a, **k), name=name)

    return [
        # the smallest run: the D2Q33 FP64 validation problem from and to numpy arrays
        named("validate_d2q33_fp64", "host", "D2Q33", "fp64", 256, 8, 1, 200, 1.5),
        # a 2D study at single precision on a grid with odd extents
        named("plane_d2q33_fp32_odd", "run", "D2Q33", "fp32", 1021, 515, 1, 40, 1.6),
        # a large 2D run in the compact form
        named("plane_d2q33_fp16", "run", "D2Q33", "fp16", 4096, 2048, 1, 20, 1.6),
        # the ordinary 3D run: a state a little larger than L2
        named("box_d3q95_fp32", "run", "D3Q95", "fp32", 128, 64, 64, 100, 1.6),
        # the benchmark's grid, FP32
        named("sweep_d3q95_fp32", "run", "D3Q95", "fp32", 512, 256, 256, 10, 1.8),
        # the benchmark's grid in the compact form, chosen where memory or speed matters most
        named("sweep_d3q95_fp16", "run", "D3Q95", "fp16", 512, 256, 256, 20, 1.8),
        # the other compact form on a ragged box that fits L2
        named("box_d3q95_bf16_ragged", "run", "D3Q95", "bf16", 250, 67, 21, 30, 1.7),
        # the FP64 form, the reference solution of a 3D precision study
        named("reference_d3q95_fp64", "run", "D3Q95", "fp64", 128, 32, 32, 20, 1.8),
        # the paper's shock tube, 11 x 11 x 800, between fixed end states
        named("tube_d3q95_fp32", "tube", "D3Q95", "fp32", 11, 11, 800, 150, 1.5),
        # continuing from populations another program produced, odd extents
        named("restart_d3q95_fp32", "restart", "D3Q95", "fp32", 201, 99, 50, 4, 1.6),
        # recovering initial fields by gradients: the adjoint benchmark's grid and spacing
        named("gradient_d3q95_fp32", "gradient", "D3Q95", "fp32", 128, 128, 128, 44, 1.6, every=22),
        # a gradient study in FP64 on a small 2D grid, omega differentiated too
        named("gradient_d2q33_fp64", "gradient", "D2Q33", "fp64", 200, 40, 1, 20, 1.5, every=5),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _extents(rng, model, cells, least=4):
    """Extents with about `cells` cells in all, x the longest as a rule, odd ones among them."""
    if model == "D2Q33":
        ny = int(max(least, _log(rng, max(least, cells ** 0.25), cells ** 0.55)))
        nx = int(max(least, cells / ny))
        nz = 1
    else:
        side = cells ** (1.0 / 3.0)
        ny = int(max(least, side * _log(rng, 0.5, 1.2)))
        nz = int(max(least, side * _log(rng, 0.5, 1.2)))
        nx = int(max(least, cells / (ny * nz)))
    if rng.random() < 0.6:              # rows that vector loads and blocks of 128 like
        m = rng.choice([8, 16, 32])
        nx = max(m, nx // m * m)
    return nx, min(ny, 65535), min(nz, 65535)


def draw(rng):
    kind = rng.choice(["host", "run", "run", "run", "run", "run", "tube", "restart", "gradient"])
    omega = round(rng.uniform(1.2, 1.85), 3)
    if kind == "host":
        model = rng.choice(["D2Q33", "D3Q95"])
        ext = _extents(rng, model, _log(rng, 1000, 30000))
        return _case(kind, model, rng.choice(["fp64", "fp32"]), *ext, rng.randint(50, 200), omega)
    if kind == "run":
        model = rng.choice(["D2Q33", "D3Q95", "D3Q95"])
        storage = rng.choice(["fp32", "fp32", "fp16", "bf16", "fp64"])
        most = 8e6 if model == "D2Q33" else 1.6e7
        if storage == "fp64":
            most = 1.3e5 if model == "D3Q95" else 1e6
        ext = _extents(rng, model, _log(rng, 5000, most))
        return _case(kind, model, storage, *ext, rng.randint(8, 20), omega)
    if kind == "tube":
        # a long thin box along z (3D) or x (2D) between two states
        n, side = int(_log(rng, 300, 2000)), rng.randint(8, 20)
        if rng.random() < 0.7:
            return _case(kind, "D3Q95", "fp32", side, side, n, rng.randint(50, 150), omega)
        return _case(kind, "D2Q33", rng.choice(["fp32", "fp64"]), n, side, 1,
                     rng.randint(50, 150), omega)
    if kind == "restart":
        model = rng.choice(["D2Q33", "D3Q95"])
        ext = _extents(rng, model, _log(rng, 1e5, 3e6 if model == "D3Q95" else 8e6))
        return _case(kind, model, rng.choice(["fp32", "fp32", "fp64"]) if model == "D2Q33" else "fp32",
                     *ext, rng.randint(2, 8), omega)
    steps = rng.randint(10, 40)
    every = max(2, int(round(math.sqrt(steps))))
    if rng.random() < 0.6:
        ext = _extents(rng, "D3Q95", _log(rng, 2e4, 2e6), least=8)
        return _case(kind, "D3Q95", "fp32", *ext, steps, omega, every=every)
    ext = _extents(rng, "D2Q33", _log(rng, 2e3, 2e4), least=8)
    return _case(kind, "D2Q33", "fp64", *ext, steps, omega, every=every)


# ------------------------------------------------------------------ velocity sets (exact, T0)
_REPS = {"D2Q33": [(0, 0), (1, 0), (1, 1), (2, 0), (2, 2), (3, 0), (2, 1), (4, 4)],
         "D3Q95": [(0, 0, 0), (2, 0, 0), (2, 2, 0), (2, 2, 2), (3, 0, 0), (3, 3, 0), (3, 3, 3),
                   (2, 2, 5), (4, 4, 0), (5, 0, 0)]}
_START = {"D2Q33": ([0.161987, 0.143204, 0.0338840, 0.00556112, 8.44799e-5, 0.00113254,
                     0.0128169, 3.45552e-6], 0.819381),
          "D3Q95": ([0.206847, 0.00442257, 0.0333341, 0.0128902, 0.0287920, 0.00264319,
                     0.000927908, 0.00106078, 0.000804376, 0.00274697], 0.421803)}
_PERMS = {2: [(0, 1), (1, 0)],
          3: [(0, 1, 2), (0, 2, 1), (1, 0, 2), (1, 2, 0), (2, 0, 1), (2, 1, 0)]}
_SETS = {}


def _velocity_set(model):
    """(e [Q, D], w [Q], c): the stored order is the rest velocity, then opposite pairs, shell
    by shell; the weights solve the paper's moment equations (Formula 5) from the printed
    digits by Newton's method."""
    if model in _SETS:
        return _SETS[model]
    D = DIM[model]
    e, grp = [(0,) * D], [0]
    for g, rep in enumerate(_REPS[model]):
        if g == 0:
            continue
        for perm in _PERMS[D]:
            for s in range(1 << D):
                v = tuple((-1 if (s >> k) & 1 else 1) * rep[perm[k]] for k in range(D))
                lead = next(x for x in v if x)
                if lead < 0 or v in e:
                    continue
                e += [v, tuple(-x for x in v)]
                grp += [g, g]
    e, grp = np.array(e), np.array(grp)
    G = grp.max() + 1
    pw = [a for a in itertools.product(range(0, 9, 2), repeat=D)
          if sum(a) <= 8 and list(a) == sorted(a, reverse=True)]
    M = np.array([[np.prod(e[grp == g].astype(float) ** np.array(a), axis=1).sum()
                   for g in range(G)] for a in pw])
    rhs = np.array([np.prod([np.prod(np.arange(k - 1, 0, -2.0)) / 2.0 ** (k // 2) for k in a])
                    for a in pw])
    deg = np.array([sum(a) for a in pw])
    W, c = np.array(_START[model][0]), _START[model][1]
    for _ in range(30):
        F = (M @ W) * c ** deg - rhs
        J = np.concatenate([M * (c ** deg)[:, None],
                            ((M @ W) * deg * c ** (deg - 1.0))[:, None]], axis=1)
        d = np.linalg.solve(J, -F)
        W, c = W + d[:-1], c + d[-1]
    _SETS[model] = (e, W[grp], float(c))
    return _SETS[model]


def _t0(model):
    return 1.0 / (2.0 * _velocity_set(model)[2] ** 2)


# ------------------------------------------------------------------ inputs
def _fields(case, seed):
    """rho [Nz, Ny, Nx], U [D, Nz, Ny, Nx], T [Nz, Ny, Nx] (lattice units), FP64 on the GPU:
    a planar Riemann problem along the longest axis, (1, 1) | (0.6, 0.75), the pair shifted and
    perturbed from the seed."""
    D, dims = DIM[case["model"]], (case["nx"], case["ny"], case["nz"])
    g = torch.Generator(device=DEVICE).manual_seed(int(seed))
    r = np.random.RandomState(int(seed) % (1 << 32))
    axis = int(np.argmax(dims))
    f64 = dict(dtype=torch.float64, device=DEVICE)
    pos = []
    for k in range(3):                          # coordinate k, broadcast over [Nz, Ny, Nx]
        shape = [1, 1, 1]
        shape[2 - k] = dims[k]
        pos.append(torch.arange(dims[k], **f64).reshape(shape))
    shape = dims[::-1]
    left = (pos[axis] < dims[axis] // 2).expand(shape)
    a = 0.02 * r.uniform(-1, 1, 2)
    rho = torch.where(left, 1.0 + a[0], 0.6 + a[0])
    T = torch.where(left, 1.0 + a[1], 0.75 + a[1])

    def wave(amp):                              # a smooth periodic perturbation
        k = r.randint(1, 3, 3)
        ph = r.uniform(0, 2 * np.pi, 3)
        v = amp
        for d in range(D):
            v = v * torch.cos(2 * np.pi * int(k[d]) * pos[d] / dims[d] + ph[d])
        return v

    rho = rho + wave(0.01) + 1e-4 * (2 * torch.rand(shape, generator=g, **f64) - 1)
    T = (T + wave(0.01)) * _t0(case["model"])
    U = torch.stack([wave(0.05).expand(shape) for _ in range(D)])
    return rho.contiguous(), U.contiguous(), T.contiguous()


def _end_states(case):
    """The tube's end states (rho, U, T) and its axis: the unperturbed sides."""
    D, t0 = DIM[case["model"]], _t0(case["model"])
    axis = int(np.argmax((case["nx"], case["ny"], case["nz"])))
    return axis, [1.0] + [0.0] * D + [t0], [0.6] + [0.0] * D + [0.75 * t0]


def prepare(case, seed):
    from paper_1303_4624_gb300 import lbm
    dims = (case["nx"], case["ny"], case["nz"])
    rho, U, T = _fields(case, seed)
    s = {"case": case, "lbm": lbm,
         "lat": lbm.Lattice(case["model"], dims, case["omega"], case["storage"])}
    kind = case["kind"]
    if kind == "host":
        s["fields"] = [a.cpu().numpy() for a in (rho, U, T)]
        return s
    if kind == "restart":
        s["f"] = _equilibrium(case["model"], rho, U, T, whole=True)
        s["out"] = torch.empty_like(s["f"])
        return s
    if kind == "gradient":
        # single-precision parameters for the FP32 form, double for FP64
        dt = torch.float32 if case["storage"] == "fp32" else torch.float64
        s["params"] = [a.to(dt).requires_grad_(True) for a in (rho, U, T)]
        s["target"] = _fields(case, seed + 1000003)[0].to(dt)
        # the FP64 study also differentiates the relaxation frequency
        s["omega"] = case["omega"]
        if case["storage"] == "fp64":
            s["omega"] = torch.tensor(case["omega"], dtype=torch.float64, requires_grad=True)
            s["params"].append(s["omega"])
        return s
    s["fields"] = [rho, U, T]
    if kind == "tube":
        axis, lo, hi = _end_states(case)
        lbm.lbm_set_fixed_ends(s["lat"].ctx, axis, 4 if case["model"] == "D2Q33" else 5, lo, hi)
    s["raw"] = torch.empty((NQ[case["model"]],) + dims[::-1], dtype=RAW[case["storage"]], device=DEVICE)
    if BYTES[case["storage"]] >= 4:
        s["moments"] = [torch.empty_like(a) for a in (rho, U, T)]
    return s


# ------------------------------------------------------------------ one pass
def run(s):
    case, lbm, lat = s["case"], s["lbm"], s["lat"]
    kind, n = case["kind"], case["steps"]
    if kind == "host":
        lat.init(*s["fields"])
        lat.step(n)
        return list(lat.moments())
    if kind == "restart":
        lbm.lbm_set_populations(lat.ctx, s["f"])
        lbm.lbm_step(lat.ctx, n)
        lbm.lbm_get_populations(lat.ctx, s["out"])
        return [s["out"]]
    if kind == "gradient":
        from paper_1303_4624_gb300.autograd import rollout
        for p in s["params"]:
            p.grad = None
        rho, U, T = s["params"][:3]
        pred = rollout(lat, rho.double(), U.double(), T.double(), s["omega"], n, case["every"])
        pred = pred.to(rho.dtype)
        loss = ((pred - s["target"]) ** 2).mean()
        loss.backward()
        return [pred.detach()] + [p.grad for p in s["params"]]
    lbm.lbm_init(lat.ctx, *s["fields"])
    lbm.lbm_step(lat.ctx, n)
    lbm.lbm_get_raw(lat.ctx, s["raw"])
    out = [s["raw"]]
    if "moments" in s:
        lbm.lbm_moments(lat.ctx, *s["moments"])
        out += s["moments"]
    return out


def work(case):
    """Bytes: the initial fields or populations read once, every population read and written
    once a step, the outputs written once; a gradient adds, for each step, one read of that
    state and one read and one write of the adjoint populations.  Flops: about 16 for each
    population of a cell update, twice that for its adjoint."""
    n = case["nx"] * case["ny"] * case["nz"]
    Q, D, b = NQ[case["model"]], DIM[case["model"]], BYTES[case["storage"]]
    fields, state, steps = (D + 2) * 8 * n, Q * b * n, case["steps"]
    flops = 16.0 * Q * n * steps
    kind = case["kind"]
    if kind == "restart":
        return {"bytes": 2.0 * 8 * Q * n + 2.0 * state * steps, "flops": flops}
    if kind == "gradient":
        adj = 3.0 * state * steps                # state and adjoint in, adjoint out
        return {"bytes": 2.0 * fields + 2.0 * state * steps + adj, "flops": 3 * flops}
    out = fields if kind == "host" else state + (fields if b >= 4 else 0)
    return {"bytes": float(fields + 2.0 * state * steps + out), "flops": flops}


# ------------------------------------------------------------------ the same in 64 bits
def _tables(model):
    e, w, c = _velocity_set(model)
    f64 = dict(dtype=torch.float64, device=DEVICE)
    xi = torch.tensor(e * (math.sqrt(2.0) * c), **f64)
    return e, torch.tensor(w, **f64), xi, (xi * xi).sum(1)


def _p_minus_1(xi, x2, u, t):
    """The Hermite polynomial of f_eq / (w rho), less one: xi [Q, D], u [D, m], t [m]."""
    D = xi.shape[1]
    q, x = (u * u).sum(0)[None], x2[:, None]
    t, s = t[None], xi @ u
    a0 = (-q / 2 + t * (x - D) / 2 +
          (3 * q * q + 6 * t * (D + 2 - x) * q + 3 * t * t * (x * x - 2 * (D + 2) * x + D * (D + 2))) / 24)
    a1 = 1 - q / 2 + t * (x - D - 2) / 2
    a2 = 0.5 - q / 4 + t * (x - D - 4) / 4
    return a0 + s * (a1 + s * (a2 + s * (1.0 / 6 + s / 24)))


def _h_eq(xi, x2, rho1, u, t):
    return rho1[None] + (1 + rho1)[None] * _p_minus_1(xi, x2, u, t)


def _chunks(n, m=1 << 18):
    return [(a, min(n, a + m)) for a in range(0, n, m)]


def _equilibrium(model, rho, U, T, whole=False):
    """Deviations h = f / w - 1 of the equilibrium of fields (populations f if whole)."""
    e, w, xi, x2 = _tables(model)
    D, n, a = xi.shape[1], rho.numel(), math.sqrt(2.0) * _velocity_set(model)[2]
    r, u, th = rho.reshape(-1), U.reshape(D, -1) * a, T.reshape(-1) / _t0(model)
    h = torch.empty((xi.shape[0], n), dtype=torch.float64, device=DEVICE)
    for i, j in _chunks(n):
        v = _h_eq(xi, x2, r[i:j] - 1, u[:, i:j], th[i:j] - 1)
        h[:, i:j] = w[:, None] * (1 + v) if whole else v
    return h.reshape((xi.shape[0],) + tuple(rho.shape))


def _state(w, xi, x2, h):
    rho1, j = w @ h, (w[:, None] * xi).T @ h
    D, rho = xi.shape[1], 1 + rho1
    u = j / rho[None]
    t = (((w * x2) @ h - D * rho1) / rho - (u * u).sum(0)) / D
    return rho1, u, t


def _collide(w, xi, x2, h, omega):
    return h + omega * (_h_eq(xi, x2, *_state(w, xi, x2, h)) - h)


def _shift(h, e, sign):
    g = torch.empty_like(h)
    for i in range(len(e)):
        v = [sign * int(x) for x in e[i]] + [0] * (3 - e.shape[1])
        g[i] = torch.roll(h[i], shifts=(v[2], v[1], v[0]), dims=(0, 1, 2))
    return g


def _advance(tab, h, omega):
    e, w, xi, x2 = tab
    g = _shift(h, e, 1)
    flat = g.reshape(g.shape[0], -1)
    for i, j in _chunks(flat.shape[1]):
        flat[:, i:j] = _collide(w, xi, x2, flat[:, i:j], omega)
    return g


def _macroscopic(model, tab, h):
    _, w, xi, x2 = tab
    flat, D, shape = h.reshape(h.shape[0], -1), xi.shape[1], tuple(h.shape[1:])
    n, a = flat.shape[1], math.sqrt(2.0) * _velocity_set(model)[2]
    rho, U, T = (torch.empty(s, dtype=torch.float64, device=DEVICE) for s in ((n,), (D, n), (n,)))
    for i, j in _chunks(n):
        r1, u, t = _state(w, xi, x2, flat[:, i:j])
        rho[i:j], U[:, i:j], T[i:j] = 1 + r1, u / a, (1 + t) * _t0(model)
    return [rho.reshape(shape), U.reshape((D,) + shape), T.reshape(shape)]


def _exact_gradient(case, seed):
    model, storage, omega, n = case["model"], case["storage"], case["omega"], case["steps"]
    tab = _tables(model)
    e, w, xi, x2 = tab
    dt = torch.float32 if storage == "fp32" else torch.float64
    fields = [a.to(dt).double() for a in _fields(case, seed)]
    target = _fields(case, seed + 1000003)[0].to(dt).double()
    states = [_equilibrium(model, *fields)]
    for _ in range(n):
        states.append(_advance(tab, states[-1], omega))
    last = states.pop()
    flat = last.reshape(last.shape[0], -1)
    rho_n = (1 + w @ flat).reshape(target.shape)
    lam = w[:, None] * (2 * (rho_n - target) / target.numel()).reshape(1, -1)
    del last, flat
    shape = (lam.shape[0],) + tuple(target.shape)
    d_om = torch.zeros((), dtype=torch.float64, device=DEVICE)
    for _ in range(n):
        g = _shift(states.pop(), e, 1).reshape(lam.shape)
        for i, j in _chunks(g.shape[1]):
            x = g[:, i:j].clone().requires_grad_(True)
            om = torch.tensor(omega, dtype=torch.float64, device=DEVICE, requires_grad=True)
            y = _collide(w, xi, x2, x, om)
            gx, go = torch.autograd.grad(y, (x, om), lam[:, i:j].contiguous())
            lam[:, i:j] = gx
            d_om += go
        lam = _shift(lam.reshape(shape), e, -1).reshape(lam.shape)
    D, a = DIM[model], math.sqrt(2.0) * _velocity_set(model)[2]
    gr = [torch.empty_like(v) for v in fields]
    r, u, th = fields[0].reshape(-1), fields[1].reshape(D, -1), fields[2].reshape(-1)
    for i, j in _chunks(r.numel()):
        leaf = [v.clone().requires_grad_(True) for v in (r[i:j], u[:, i:j], th[i:j])]
        h = _h_eq(xi, x2, leaf[0] - 1, leaf[1] * a, leaf[2] / _t0(model) - 1)
        got = torch.autograd.grad(h, leaf, lam[:, i:j].contiguous())
        gr[0].reshape(-1)[i:j], gr[1].reshape(D, -1)[:, i:j], gr[2].reshape(-1)[i:j] = got
    return [rho_n] + gr + ([d_om] if storage == "fp64" else [])


def exact(case, seed):
    kind, model, omega = case["kind"], case["model"], case["omega"]
    if kind == "gradient":
        return _exact_gradient(case, seed)
    tab = _tables(model)
    w = tab[1].reshape(-1, 1, 1, 1)
    rho, U, T = _fields(case, seed)
    h = _equilibrium(model, rho, U, T)
    ends = None
    if kind == "tube":
        axis, lo, hi = _end_states(case)
        D, width = DIM[model], 4 if model == "D2Q33" else 5
        ends = []
        for st, sl in ((lo, slice(0, width)), (hi, slice(-width, None))):
            v = [torch.tensor(x, dtype=torch.float64, device=DEVICE) for x in (st[0], st[1:1 + D], st[-1])]
            at = [slice(None)] * 4
            at[3 - axis] = sl
            ends.append((tuple(at), _equilibrium(model, v[0].reshape(1, 1, 1), v[1].reshape(D, 1, 1, 1),
                                                 v[2].reshape(1, 1, 1))))
    for _ in range(case["steps"]):
        h = _advance(tab, h, omega)
        for at, v in ends or ():
            h[at] = v
    if kind == "host":
        return _macroscopic(model, tab, h)
    if kind == "restart":
        return [w * (1 + h)]
    out = [h]
    if BYTES[case["storage"]] >= 4:
        out += _macroscopic(model, tab, h)
    return out
