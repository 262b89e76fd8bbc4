"""The work that programs have this library do, as cases to time and to compare.

A case is one call sequence of such a program through `binding.SPH` (or
`sph_conserved_noalloc`), on inputs made on the GPU from a seed: the rotating
square patch at the sizes the benchmark and the tests use it (20^3 to 200^3)
with its lattice lightly disturbed, the irregular patch (jittered lattice,
log-normal masses, 50-400 neighbours), and batches of independent patches.
Kinds:

  run       a short simulation from given particles: set_particles, steps,
            the new state read back (latency decides at these sizes); mixed
            runs keep h, whose adaptation turns on whole neighbour counts
            that an FP32 rounding can change
  step      one step at the sizes of production runs, h adapting
  batch     a run of many patches of uneven size advanced together
  search    one neighbour search, with its counts |N(i)| and n_i
  lists     one neighbour search, with the lists themselves
  forces    density, pressure, accelerations and du/dt on given lists
  conserved the conserved sums of arrays the caller holds

The mixed path sums in FP32: its densities and forces are FP32 values, and the
velocities and energies it steps carry FP32 forces, so they are returned as
float32; the FP64 path's results are float64 and counts are whole numbers.
"""
import math

import numpy as np
import torch

from paper_1905_03344_gb300 import binding, inputs

DEV = "cuda"
GAMMA, COURANT, GROWTH, N_TARGET = 5.0 / 3.0, 0.2, 1.1, 100.0
ALPHA, BETA, EPS = 1.0, 2.0, 0.01


def listed():
    return [
        # the smallest configuration in use: 8000 particles, FP64, ten steps
        {"name": "run_20_fp64", "kind": "run", "edge": 20, "precision": "fp64", "steps": 10, "adapt_h": 1},
        # a small mixed run of odd size, h frozen (a parameter sweep's member)
        {"name": "run_33_mixed", "kind": "run", "edge": 33, "precision": "mixed", "steps": 10, "adapt_h": 0},
        # lists handed to other code (analysis, another solver)
        {"name": "lists_45", "kind": "lists", "edge": 45, "spread": 0.0, "irregular": False},
        # the paper's million particles well into a run: h has grown behind
        # the free surface
        {"name": "search_100", "kind": "search", "edge": 100, "spread": 0.35, "irregular": False},
        # the pair sums of the paper's million particles, default launch shape
        {"name": "forces_100", "kind": "forces", "edge": 100, "spread": 0.35, "irregular": False,
         "precision": "mixed", "kernel": "wendland", "grad_h": 0, "pair_bins": 0},
        # uneven rows: every particle its own h
        {"name": "search_irregular_80", "kind": "search", "edge": 80, "spread": 0.0, "irregular": True},
        # ... and their sums, balanced by row-length bins
        {"name": "forces_irregular_80", "kind": "forces", "edge": 80, "spread": 0.0, "irregular": True,
         "precision": "mixed", "kernel": "wendland", "grad_h": 0, "pair_bins": 32},
        # the reference-precision path
        {"name": "forces_50_fp64", "kind": "forces", "edge": 50, "spread": 0.0, "irregular": False,
         "precision": "fp64", "kernel": "wendland", "grad_h": 0, "pair_bins": 0},
        # the second kernel with the grad-h form
        {"name": "forces_63_sinc_gradh", "kind": "forces", "edge": 63, "spread": 0.0, "irregular": False,
         "precision": "mixed", "kernel": "sinc", "grad_h": 1, "pair_bins": 0},
        # diagnostics of a host framework's own arrays
        {"name": "conserved_2m", "kind": "conserved", "n": 2000003},
        # 64 independent patches, edges 10 to 60, replayed as a CUDA graph
        {"name": "batch_64", "kind": "batch", "count": 64, "lo": 10, "hi": 60, "steps": 5, "adapt_h": 0},
        # the headline size, in the launch shape the autotuner settles on there
        {"name": "step_200", "kind": "step", "edge": 200, "precision": "mixed", "steps": 1,
         "adapt_h": 1, "lanes": 2},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["run", "run", "lists", "search", "search", "forces", "forces", "forces", "conserved", "batch",
                       "step"])
    if kind == "run":
        prec = rng.choice(["fp64", "mixed"])
        return {"kind": kind, "edge": rng.randint(10, 34), "precision": prec, "steps": rng.randint(5, 12),
                "adapt_h": int(prec == "fp64")}
    if kind == "lists":
        return {"kind": kind, "edge": _log(rng, 12, 64), "spread": rng.choice([0.0, 0.35]),
                "irregular": rng.random() < 0.3}
    if kind == "search":
        irr = rng.random() < 0.4
        return {"kind": kind, "edge": _log(rng, 20, 80 if irr else 120), "spread": 0.0 if irr else rng.choice([0.0, 0.35]),
                "irregular": irr}
    if kind == "forces":
        irr = rng.random() < 0.35
        prec = rng.choice(["mixed", "mixed", "fp64"])
        kern = rng.choice(["wendland", "wendland", "sinc"])
        hi = 64 if prec == "fp64" else (80 if irr else 110)
        return {"kind": kind, "edge": _log(rng, 20, hi), "spread": 0.0 if irr else rng.choice([0.0, 0.35]),
                "irregular": irr, "precision": prec, "kernel": kern, "grad_h": int(rng.random() < 0.3),
                "pair_bins": rng.choice([32, 64]) if irr else 0}
    if kind == "conserved":
        return {"kind": kind, "n": _log(rng, 1000, 8000000) | 1}
    if kind == "batch":
        lo = rng.randint(10, 16)
        return {"kind": kind, "count": rng.randint(5, 48), "lo": lo, "hi": rng.randint(lo + 5, 56), "steps": 3,
                "adapt_h": 0}
    return {"kind": kind, "edge": _log(rng, 50, 180), "precision": "mixed", "steps": 1, "adapt_h": 1,
            "lanes": rng.choice([0, 2])}


# ---- inputs --------------------------------------------------------------------
def _layer_u(n, omega):
    """Specific internal energy of one lattice layer (n^2 values) from the patch's pressure."""
    g = inputs.lattice_1d(n)
    yy, xx = np.meshgrid(g, g, indexing="ij")
    p = inputs.pressure_series(xx.ravel(), yy.ravel(), omega, nmax=59 if n < 64 else 199)
    return (p + inputs.pressure_offset(omega)) / (GAMMA - 1.0)


def _patch(n, gen, irregular=False, spread=0.0, omega=(4.5, 5.5)):
    """A square patch of n^3 particles as float64 tensors on the GPU."""
    kw = dict(generator=gen, dtype=torch.float64, device=DEV)
    dx, N = 1.0 / n, n ** 3
    omega = omega[0] + (omega[1] - omega[0]) * float(torch.rand((), **kw))
    g = torch.as_tensor(inputs.lattice_1d(n), device=DEV)
    z, y, x = (t.reshape(-1).clone() for t in torch.meshgrid(g, g, g, indexing="ij"))
    sig = (0.3 if irregular else 0.04) * dx
    for t in (x, y, z):
        t += sig * torch.randn(N, **kw).clamp_(-5.0, 5.0)
    z -= torch.floor(z + 0.5)
    z[z >= 0.5] -= 1.0
    m = torch.full((N,), 1.0 / N, dtype=torch.float64, device=DEV)
    h = torch.full((N,), inputs.ETA * dx, dtype=torch.float64, device=DEV)
    if irregular:
        f = torch.exp(0.5 * torch.randn(N, **kw))
        m *= f
        h *= f ** (1.0 / 3.0)
    if spread > 0.0:
        # h behind the free surface, where half (or three quarters, at the
        # edges) of the neighbours are missing
        for t in (x, y):
            h *= 1.0 + spread * torch.exp(-(0.5 - t.abs()).clamp_min(0.0) / (2.0 * dx))
    u = torch.as_tensor(_layer_u(n, omega), device=DEV).repeat(n)
    return {"x": x, "y": y, "z": z, "vx": omega * y, "vy": -omega * x, "vz": 0.05 * torch.randn(N, **kw),
            "m": m, "h": h, "u": u}


def _edges(case):
    """Lattice edges of a batch's patches: part of the case, the same for every seed."""
    return np.random.default_rng(case["count"]).integers(case["lo"], case["hi"] + 1, case["count"])


def _fields(case, seed):
    gen = torch.Generator(device=DEV).manual_seed(int(seed))
    kind = case["kind"]
    if kind == "conserved":
        kw = dict(generator=gen, dtype=torch.float64, device=DEV)
        n = case["n"]
        f = {k: torch.rand(n, **kw) - 0.5 for k in ("x", "y")}
        f.update({k: 3.0 * torch.randn(n, **kw) for k in ("vx", "vy", "vz")})
        f["m"] = (0.5 + torch.rand(n, **kw)) / n
        f["u"] = 1000.0 + 100.0 * torch.rand(n, **kw)
        return f, None
    if kind == "batch":
        edges = _edges(case)
        parts = [_patch(int(e), gen, omega=(2.0, 8.0)) for e in edges]
        f = {k: torch.cat([p[k] for p in parts]) for k in parts[0]}
        off = np.zeros(len(edges) + 1, dtype=np.int64)
        off[1:] = np.cumsum(edges.astype(np.int64) ** 3)
        return f, off
    return _patch(case["edge"], gen, case.get("irregular", False), case.get("spread", 0.0)), None


def prepare(case, seed):
    f, off = _fields(case, seed)
    s = {"case": case, "f": f, "off": off}
    if case["kind"] == "conserved":
        s["out"] = torch.zeros(7, dtype=torch.float64, device=DEV)
        torch.cuda.synchronize()
        return s
    n = len(f["x"])
    opt = {}
    if case["kind"] == "forces":
        opt = {"kernel": case["kernel"], "grad_h": case["grad_h"], "pair_bins": case["pair_bins"]}
    if "adapt_h" in case:
        opt["adapt_h"] = case["adapt_h"]
    if case.get("lanes"):
        opt["threads_per_particle"] = case["lanes"]
    if off is not None:
        opt["use_graph"] = 1
    s["n"] = n
    s["stream"] = torch.cuda.Stream()
    s["sim"] = binding.SPH(n, precision=case.get("precision", "mixed"), max_patches=1 if off is None else len(off) - 1,
                           stream=s["stream"].cuda_stream, **opt)
    torch.cuda.synchronize()
    if case["kind"] in ("search", "lists", "forces"):
        s["sim"].set_particles(f)
    if case["kind"] == "forces":
        s["sim"].find_neighbors()
    if case["kind"] == "lists":
        # buffers for the lists, as large as the library's own default capacity
        s["off"] = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
        s["col"] = torch.zeros(160 * n, dtype=torch.int32, device=DEV)
        s["perm"] = torch.zeros(n, dtype=torch.int32, device=DEV)
        torch.cuda.synchronize()
    return s


def _read(s, names):
    out = torch.empty(len(names), s["n"], dtype=torch.float64, device=DEV)
    for k, name in enumerate(names):
        s["sim"].field(name, out=out[k])
    return out


def run(s):
    case = s["case"]
    if case["kind"] == "conserved":
        binding.sph_conserved_noalloc(s["f"], s["out"], torch.cuda.current_stream().cuda_stream)
        return s["out"]
    sim = s["sim"]
    cast = (lambda t: t) if case.get("precision") == "fp64" else (lambda t: t.float())
    with torch.cuda.stream(s["stream"]):
        if case["kind"] in ("search", "lists"):
            sim.find_neighbors()
            if case["kind"] == "lists":
                buf = [s[k] for k in ("off", "col", "perm")]
                binding._check(sim.ctx, binding.lib().sph_copy_neighbors(sim.ctx, *(t.data_ptr() for t in buf), 1))
                return buf
            return {"nnb": _read(s, ["nnb"]).long(), "nown": _read(s, ["nown"]).long()}
        if case["kind"] == "forces":
            sim.density()
            sim.momentum_energy()
            return {k: cast(_read(s, v)) for k, v in (("rho", ["rho"]), ("P", ["P"]), ("c", ["c"]),
                                                      ("a", ["ax", "ay", "az"]), ("du", ["du"]))}
        sim.set_particles(s["f"])
        if s["off"] is not None:
            sim.set_patches(s["off"])
        dt = sim.step(case["steps"])
        out = {k: cast(_read(s, v)) for k, v in (("x", ["x", "y", "z"]), ("v", ["vx", "vy", "vz"]), ("u", ["u"]),
                                                 ("h", ["h"]), ("rho", ["rho"]), ("a", ["ax", "ay", "az"]),
                                                 ("du", ["du"]))}
        out["dt"] = dt
        return out


# ---- the least each path can do --------------------------------------------------
def work(case):
    kind = case["kind"]
    if kind == "conserved":
        return {"bytes": 56.0 * case["n"] + 56.0, "flops": 24.0 * case["n"]}
    if kind == "batch":
        edges = _edges(case)
        n = float((edges.astype(np.int64) ** 3).sum())
    else:
        n = float(case["edge"]) ** 3
    # neighbours of a particle: about 100, more where h varies (the union)
    nb = 150.0 if case.get("irregular") else 105.0
    size = 8.0 if case.get("precision") == "fp64" else 4.0
    if kind == "search":
        return {"bytes": n * (32.0 + 16.0) + 4.0 * n * nb, "flops": 8.0 * n * nb}
    if kind == "lists":
        return {"bytes": n * (32.0 + 12.0) + 4.0 * n * nb, "flops": 8.0 * n * nb}
    pair = {"wendland": 28.0 + 70.0, "sinc": 40.0 + 92.0}[case.get("kernel", "wendland")]
    if kind == "forces":
        return {"bytes": n * (9.0 * size + 4.0 * nb + 7.0 * size), "flops": pair * n * nb}
    # a step reads the particle state and writes it, and its forces, once
    return {"bytes": case["steps"] * n * (13.0 * 8.0 * 2.0 + 5.0 * size), "flops": case["steps"] * n * nb * (8.0 + pair)}


# ---- the same results in plain 64-bit torch ---------------------------------------
def _pairs(f, lz=1.0):
    """Blocks (rows, idx, valid): candidates idx[r, k] of the particles rows, every
    pair within 2 max h among them once; valid masks the padding and j = i."""
    n = len(f["x"])
    dev = f["x"].device
    ar = torch.arange(n, device=dev)
    big = 1 << 25
    if n <= 40000:
        c = max(1, big // n)
        for a in range(0, n, c):
            rows = ar[a:a + c]
            idx = ar.expand(len(rows), n)
            yield rows, idx, idx != rows[:, None]
        return
    edge = 2.0 * float(f["h"].max()) * (1.0 + 1e-9)
    x0, y0 = f["x"].min(), f["y"].min()
    nx = max(1, int(float(f["x"].max() - x0) / edge))
    ny = max(1, int(float(f["y"].max() - y0) / edge))
    nz = max(1, int(lz / edge))
    ex, ey, ez = float(f["x"].max() - x0) / nx, float(f["y"].max() - y0) / ny, lz / nz
    cx = ((f["x"] - x0) / ex).long().clamp_(0, nx - 1)
    cy = ((f["y"] - y0) / ey).long().clamp_(0, ny - 1)
    cz = ((f["z"] + 0.5 * lz) / ez).long().clamp_(0, nz - 1)
    key = (cz * ny + cy) * nx + cx
    order = torch.argsort(key)
    cnt = torch.bincount(key, minlength=nx * ny * nz)
    start = torch.cumsum(cnt, 0) - cnt
    M = int(cnt.max())
    k = torch.arange(M, device=dev)
    zoff = range(-1, 2) if nz >= 3 else range(nz)
    c = max(1, big // M)
    for a in range(0, n, c):
        rows = order[a:a + c]
        for dz in zoff:
            zz = (cz[rows] + dz) % nz
            for dy in (-1, 0, 1):
                yy = cy[rows] + dy
                for dx in (-1, 0, 1):
                    xx = cx[rows] + dx
                    ok = (yy >= 0) & (yy < ny) & (xx >= 0) & (xx < nx)
                    cell = ((zz * ny + yy.clamp(0, ny - 1)) * nx + xx.clamp(0, nx - 1))
                    valid = ok[:, None] & (k[None, :] < cnt[cell][:, None])
                    idx = order[(start[cell][:, None] + k[None, :]).clamp_(max=n - 1)]
                    yield rows, idx, valid & (idx != rows[:, None])


def _sep(f, rows, idx, lz=1.0):
    dx = f["x"][rows][:, None] - f["x"][idx]
    dy = f["y"][rows][:, None] - f["y"][idx]
    dz = f["z"][rows][:, None] - f["z"][idx]
    dz = torch.where(dz > 0.5 * lz, dz - lz, torch.where(dz < -0.5 * lz, dz + lz, dz))
    return dx, dy, dz, (dx * dx + dy * dy) + dz * dz


def _near(f, rows, idx, valid, r2):
    own = valid & (r2 < ((4.0 * f["h"]) * f["h"])[rows][:, None])
    return own, own | (valid & (r2 < ((4.0 * f["h"]) * f["h"])[idx]))


def _sinc_norm(n):
    v, w = np.polynomial.legendre.leggauss(400)
    v, w = v + 1.0, w
    return 1.0 / (4.0 * math.pi * float((w * v * v * np.sinc(0.5 * v) ** n).sum()))


def _sinc_g(x):
    """(sin x - x cos x) / x^3, by its series near 0."""
    x2 = x * x
    t = torch.zeros_like(x)
    fact, pw = 6.0, torch.ones_like(x)
    for k in range(1, 11):
        t = t + (2.0 * k * (1.0 if k % 2 else -1.0) / fact) * pw
        pw = pw * x2
        fact *= (2.0 * k + 2.0) * (2.0 * k + 3.0)
    xs = torch.where(x < 1.0, torch.ones_like(x), x)
    return torch.where(x < 1.0, t, (torch.sin(xs) - xs * torch.cos(xs)) / (xs * xs * xs))


def _shape(kernel, r, w, n=6):
    """The kernel's r-dependent factors: S(v), -(dS/dr)/r / w^2 and -v S'(v), zero past the support (w = 1/2h)."""
    if kernel == "wendland":
        q = (1.0 - r * w).clamp_min(0.0)
        return q ** 4 * (5.0 - 4.0 * q), 20.0 * q ** 3, 20.0 * (1.0 - q) ** 2 * q ** 3
    x = math.pi * r * w
    inside = x < math.pi
    x = torch.where(inside, x, torch.zeros_like(x))
    s = torch.sinc(x / math.pi)
    g = _sinc_g(x)
    z = torch.zeros_like(x)
    return (torch.where(inside, s ** n, z), torch.where(inside, n * math.pi ** 2 * s ** (n - 1) * g, z),
            torch.where(inside, n * s ** (n - 1) * x * x * g, z))


def _forces(f, vh, kernel="wendland", grad_h=0):
    """n_i, rho, P, c, a, du of fields f, the viscosity with the velocities vh."""
    n = len(f["x"])
    kb = 21.0 / (16.0 * math.pi) if kernel == "wendland" else _sinc_norm(6)
    w = 0.5 / f["h"]
    zero = lambda: torch.zeros(n, dtype=torch.float64, device=f["x"].device)  # noqa: E731
    sd, so, nown = zero(), zero(), zero()
    for rows, idx, valid in _pairs(f):
        _, _, _, r2 = _sep(f, rows, idx)
        own, near = _near(f, rows, idx, valid, r2)
        nown.index_add_(0, rows, own.sum(1).double())
        s, _, o = _shape(kernel, torch.sqrt(r2), w[rows][:, None])
        m = f["m"][idx] * near
        sd.index_add_(0, rows, (m * s).sum(1))
        if grad_h:
            so.index_add_(0, rows, (m * o).sum(1))
    rho = kb / f["h"] ** 3 * (f["m"] + sd)
    P = (GAMMA - 1.0) * rho * f["u"]
    c = torch.sqrt(GAMMA * P / rho)
    A = P / (rho * rho)
    if grad_h:
        A = A / (so / (3.0 * (f["m"] + sd)))
    acc, du = torch.zeros(3, n, dtype=torch.float64, device=f["x"].device), zero()
    for rows, idx, valid in _pairs(f):
        dx, dy, dz, r2 = _sep(f, rows, idx)
        _, near = _near(f, rows, idx, valid, r2)
        r = torch.sqrt(r2)
        R = lambda t: t[rows][:, None]  # noqa: E731
        # grad_i W(r, h) = -kb/h^3 w^2 G(r) (x_i - x_j)
        gi = R(kb / f["h"] ** 3 * w * w) * _shape(kernel, r, R(w))[1]
        gj = (kb / f["h"] ** 3 * w * w)[idx] * _shape(kernel, r, w[idx])[1]
        vx, vy, vz = (R(v) - v[idx] for v in vh)
        vd = vx * dx + vy * dy + vz * dz
        hb = 0.5 * (R(f["h"]) + f["h"][idx])
        mu = hb * vd / (r2 + EPS * hb * hb)
        pi = (-ALPHA * 0.5 * (R(c) + c[idx]) * mu + BETA * mu * mu) / (0.5 * (R(rho) + rho[idx]))
        pi = torch.where(vd < 0.0, pi, torch.zeros_like(pi))
        m = f["m"][idx] * near
        gb = 0.5 * (gi + gj)
        if grad_h:
            fa = m * (R(A) * gi + A[idx] * gj + pi * gb)
            fu = m * (R(A) * gi + 0.5 * pi * gb)
        else:
            fa = m * (R(A) + A[idx] + pi) * gb
            fu = m * (R(A) + 0.5 * pi) * gb
        for q, d in enumerate((dx, dy, dz)):
            acc[q].index_add_(0, rows, (fa * d).sum(1))
        du.index_add_(0, rows, (-fu * vd).sum(1))
    return {"nown": nown, "rho": rho, "P": P, "c": c, "a": acc, "du": du}


def exact(case, seed):
    kind = case["kind"]
    if kind in ("batch", "step", "lists"):
        return None
    f, _ = _fields(case, seed)
    if kind == "conserved":
        x, y, vx, vy, vz, m, u = (f[k] for k in ("x", "y", "vx", "vy", "vz", "m", "u"))
        return torch.stack([m.sum(), (m * vx).sum(), (m * vy).sum(), (m * vz).sum(), (m * (x * vy - y * vx)).sum(),
                            (0.5 * m * (vx * vx + vy * vy + vz * vz)).sum(), (m * u).sum()])
    if kind == "search":
        n = len(f["x"])
        nnb, nown = (torch.zeros(n, dtype=torch.int64, device=DEV) for _ in range(2))
        for rows, idx, valid in _pairs(f):
            own, near = _near(f, rows, idx, valid, _sep(f, rows, idx)[3])
            nnb.index_add_(0, rows, near.sum(1))
            nown.index_add_(0, rows, own.sum(1))
        return {"nnb": nnb[None], "nown": nown[None]}
    v = [f["vx"], f["vy"], f["vz"]]
    if kind == "forces":
        r = _forces(f, v, case["kernel"], case["grad_h"])
        return {"rho": r["rho"][None], "P": r["P"][None], "c": r["c"][None], "a": r["a"], "du": r["du"][None]}
    dt_prev, du_prev = 0.0, torch.zeros_like(f["u"])
    ap = torch.zeros(3, len(f["x"]), dtype=torch.float64, device=DEV)
    for k in range(case["steps"]):
        vh = [f[q] + 0.5 * dt_prev * ap[i] for i, q in enumerate(("vx", "vy", "vz"))]
        r = _forces(f, vh)
        dt = COURANT * float((f["h"] / r["c"]).min())
        if k:
            dt = min(dt, GROWTH * dt_prev)
        for i, (p, q) in enumerate((("x", "vx"), ("y", "vy"), ("z", "vz"))):
            f[q] = f[q] + r["a"][i] * (0.5 * (dt + dt_prev))
            f[p] = f[p] + f[q] * dt
        f["z"] = torch.where(f["z"] >= 0.5, f["z"] - 1.0, torch.where(f["z"] < -0.5, f["z"] + 1.0, f["z"]))
        e = 0.5 * dt / dt_prev if k else 0.0
        f["u"] = f["u"] + dt * ((1.0 + e) * r["du"] - e * du_prev)
        if case["adapt_h"]:
            f["h"] = f["h"] * torch.where(r["nown"] > 0, 0.5 * (1.0 + (N_TARGET / r["nown"].clamp_min(1.0)) ** (1.0 / 3.0)), 2.0)
        dt_prev, du_prev, ap = dt, r["du"], r["a"]
    return {"x": torch.stack([f["x"], f["y"], f["z"]]), "v": torch.stack([f["vx"], f["vy"], f["vz"]]), "u": f["u"][None],
            "h": f["h"][None], "rho": r["rho"][None], "a": r["a"], "du": r["du"][None], "dt": torch.tensor(dt, dtype=torch.float64)}
