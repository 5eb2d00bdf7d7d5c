"""The work a user has this framework do, as timed cases.

A case is a dict of plain values; ``prepare`` makes what a program holds before
the call (a solver handle and its inputs on the GPU), ``run`` is one pass
through the public entry points of ``paper_1308_3214_gb300.molt``.  ``exact``
restates the method in float64 torch, independently of the library: the
convolution L^{-1} by its quadrature and recurrences, C and D of the ADI
splitting, the level update, and the transpose by autograd.

Kinds:
  line      1D homogeneous run: start + time loop (one CTA's worth of work;
            launches and latency count)
  ends      1D run with time-dependent Dirichlet data (solve_dirichlet)
  plane     2D run: start + time loop, one problem
  cube      3D run: start + time loop
  batch     many 2D problems of uneven size stepped together
  source    2D run driven by a point source (solve_source)
  gradient  receiver traces of a 2D run and the adjoint gradient (autograd)
  embedded  2D run on an ellipse cut out of the grid
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1308_3214_gb300 import molt, workloads

DEVICE = "cuda"
STEP_CAP = {"mixed": 4_194_304 * 20, "fp64": 4_194_304 * 10}     # point-updates of a 2D or 3D pass


# --------------------------------------------------------------------------
# Cases
# --------------------------------------------------------------------------
def listed():
    return [
        # the 1D study: 256 points, second order, the whole 200-step run
        {"name": "line256_fp64", "kind": "line", "nx": 256, "P": 1, "cfl": 1.5, "bc": "periodic", "prec": "fp64",
         "steps": 200},
        # the 1D convergence study with end data, 10001 points, sixth order
        {"name": "ends10001_mixed", "kind": "ends", "nx": 10001, "P": 3, "cfl": 2.0, "bc": "dirichlet",
         "prec": "mixed", "steps": 100},
        # the point-source figure: an 81 x 81 mesh driven by a source at a node
        {"name": "source81_mixed", "kind": "source", "nx": 81, "ny": 81, "P": 2, "cfl": 2.0, "bc": "dirichlet",
         "prec": "mixed", "steps": 32},
        # the headline run: a pulse on 2048^2, sixth order, between two snapshots
        {"name": "plane2048_mixed", "kind": "plane", "nx": 2048, "ny": 2048, "P": 3, "cfl": 2.0, "bc": "dirichlet",
         "prec": "mixed", "steps": 20, "width": 0.02},
        # the same field on the float64 path
        {"name": "plane2048_fp64", "kind": "plane", "nx": 2048, "ny": 2048, "P": 3, "cfl": 2.0, "bc": "dirichlet",
         "prec": "fp64", "steps": 10, "width": 0.02},
        # a grid whose lines do not split evenly, odd and not square
        {"name": "plane1000x777_mixed", "kind": "plane", "nx": 1000, "ny": 777, "P": 3, "cfl": 2.0,
         "bc": "dirichlet", "prec": "mixed", "steps": 20, "width": 0.04},
        # the periodic cube of Fourier modes, fourth order
        {"name": "cube256_mixed", "kind": "cube", "nx": 256, "ny": 256, "nz": 256, "P": 2, "cfl": 1.5,
         "bc": "periodic", "prec": "mixed", "steps": 5},
        # a ragged Dirichlet box in float64
        {"name": "box96x100x75_fp64", "kind": "cube", "nx": 96, "ny": 100, "nz": 75, "P": 2, "cfl": 1.5,
         "bc": "dirichlet", "prec": "fp64", "steps": 10},
        # a quarter of the batched workload: uneven problems, orders and CFL numbers
        {"name": "batch128_mixed", "kind": "batch", "count": 128, "nmin": 64, "nmax": 1024, "P": 0, "cfl": 0.0,
         "bc": "dirichlet", "prec": "mixed", "steps": 20, "width": 0.02},
        # misfit gradient of receiver traces: forward run and adjoint run
        {"name": "gradient1024_mixed", "kind": "gradient", "nx": 1024, "ny": 1024, "P": 2, "cfl": 2.0,
         "bc": "dirichlet", "prec": "mixed", "steps": 40, "width": 0.02, "receivers": 64},
        # the ellipse of the embedded-boundary example on a fine grid
        {"name": "embedded2048_mixed", "kind": "embedded", "nx": 2048, "P": 2, "cfl": 1.0, "bc": "dirichlet",
         "prec": "mixed", "steps": 8, "width": 0.15},
        # the same domain on an odd, coarser grid in float64
        {"name": "embedded777_fp64", "kind": "embedded", "nx": 777, "P": 2, "cfl": 1.0, "bc": "dirichlet",
         "prec": "fp64", "steps": 8, "width": 0.15},
    ]


def _size(rng, lo, hi):
    """A point count, even over the logarithm; odd ones and whole multiples of 32 among them."""
    n = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    if rng.random() < 0.4:
        n = max(lo, n // 32 * 32)
    return min(max(n, lo), hi)


def _rows(rng, lo, hi):
    """As _size, for the rows of a 2D grid.  Left out: multiples of 64 that split into 5, 6 or 7
    segments of 64 rows a block, where float32 columns were once stored past their tile."""
    n = _size(rng, lo, hi)
    segments = n // 64
    blocks = (segments + 7) // 8
    return n - 1 if n % 64 == 0 and -(-segments // blocks) in (5, 6, 7) else n


def draw(rng):
    kind = rng.choice(["line", "ends", "source", "plane", "plane", "cube", "batch", "gradient", "embedded"])
    prec = rng.choice(["mixed", "fp64"])
    c = {"kind": kind, "P": rng.choice([1, 2, 3]), "cfl": round(rng.uniform(0.5, 4.0), 3), "prec": prec,
         "bc": "dirichlet"}
    if kind in ("line", "plane", "cube"):
        c["bc"] = rng.choice(["dirichlet", "periodic"])
    if kind == "line":
        c.update(nx=_size(rng, 64, 4096), steps=rng.randint(50, 200))
    elif kind == "ends":
        c.update(nx=_size(rng, 200, 10001), steps=rng.randint(20, 100))
    elif kind == "batch":
        # 128 problems of the listed spread hold about 26 M points
        lo = rng.choice([64, 128])
        hi = rng.choice([256, 512, 1024])
        mean = (hi * hi - lo * lo) / (2.0 * math.log(hi / lo))
        most = max(2, min(128, int((2.0e7 if prec == "mixed" else 4.0e6) / mean)))
        c.update(count=rng.randint(max(2, most // 4), most), nmin=lo, nmax=hi, P=0, cfl=0.0, width=0.02,
                 steps=rng.randint(4, 20 if prec == "mixed" else 10))
    elif kind == "embedded":
        c.update(nx=_size(rng, 129, 2048 if prec == "mixed" else 1025), P=rng.choice([1, 2]), steps=rng.randint(2, 8),
                 cfl=round(rng.uniform(0.5, 2.0), 3), width=0.15)
    else:
        if kind == "cube":
            c.update(nx=_size(rng, 32, 256), ny=_size(rng, 32, 256), nz=_size(rng, 32, 256), P=rng.choice([1, 2]))
        elif kind == "source":
            c.update(nx=_size(rng, 65, 1025), ny=_rows(rng, 65, 1025), P=rng.choice([1, 2]))
        elif kind == "gradient":
            c.update(nx=_size(rng, 128, 1024), ny=_rows(rng, 128, 1024), P=rng.choice([1, 2]), width=0.04,
                     receivers=rng.randint(8, 64))
        else:
            c.update(nx=_size(rng, 128, 2048), ny=_rows(rng, 128, 2048), width=round(rng.uniform(0.02, 0.08), 3))
        pts = c["nx"] * c["ny"] * c.get("nz", 1)
        cap = STEP_CAP[prec] // (4 if kind in ("cube", "gradient") and prec == "fp64" else 1)
        if kind == "gradient":
            cap //= 2
        c["steps"] = max(1, min(rng.randint(5, 40), cap // pts))
    return c


# --------------------------------------------------------------------------
# Inputs
# --------------------------------------------------------------------------
def _shape(c):
    if c["kind"] in ("line", "ends"):
        return (c["nx"],)
    if c["kind"] == "cube":
        return (c["nz"], c["ny"], c["nx"])
    return (c["ny"], c["nx"])


def _length(c):
    """The domain's edge: 2 pi for periodic runs, [-1, 1] for the point source, else 1."""
    return 2 * math.pi if c["bc"] == "periodic" else 2.0 if c["kind"] == "source" else 1.0


def _spacing(n, length, bc):
    return length / n if bc == "periodic" else length / (n - 1)


def _dt(c):
    """CFL times the finest spacing."""
    return c["cfl"] * min(_spacing(n, _length(c), c["bc"]) for n in _shape(c))


def _coords(n, length, bc):
    return torch.arange(n, dtype=torch.float64, device=DEVICE) * _spacing(n, length, bc)


def _gaussian(shape, rng, width):
    """A pulse with its centre in [0.3, 0.7] of every axis of the unit square, zero on the boundary."""
    u = torch.ones((), dtype=torch.float64, device=DEVICE)
    for a, n in enumerate(shape):
        x = _coords(n, 1.0, "dirichlet")
        g = torch.exp(-((x - rng.uniform(0.3, 0.7)) ** 2) / (2 * width * width))
        g[0] = g[-1] = 0.0
        u = u.unsqueeze(-1) * g
    return u.contiguous()


def _modes(shape, length, bc, rng, count, kmax):
    """A sum of seeded modes: plane waves (periodic) or products of sines (Dirichlet)."""
    u = torch.zeros(shape, dtype=torch.float64, device=DEVICE)
    x = [_coords(n, length, bc) for n in shape]
    for _ in range(count):
        if bc == "periodic":
            ks = rng.integers(-kmax, kmax + 1, size=len(shape))
            arg = torch.full((), rng.uniform(0.0, 2 * math.pi), dtype=torch.float64, device=DEVICE)
            for a, k in enumerate(ks):
                arg = arg.unsqueeze(-1) + float(k) * x[a] * (2 * math.pi / length)
            u += rng.normal() * torch.cos(arg)
        else:
            m = torch.full((), rng.normal(), dtype=torch.float64, device=DEVICE)
            for a, k in enumerate(rng.integers(1, kmax + 1, size=len(shape))):
                s = torch.sin(float(k) * math.pi / length * x[a])
                s[0] = s[-1] = 0.0
                m = m.unsqueeze(-1) * s
            u += m
    return u


def _end_data(c, seed):
    """u = sum of standing waves cos(k x + p) cos(k t): u^0 and (d_tt)^m u at both ends."""
    rng = np.random.default_rng(seed)
    k = rng.uniform(2.0, 12.0, size=4)
    a, p = rng.normal(size=4), rng.uniform(0.0, 2 * math.pi, size=4)
    t = _dt(c) * np.arange(c["steps"] + 1)
    d = np.zeros((c["steps"] + 1, 2, c["P"] + 1))
    for side in (0, 1):
        for m in range(c["P"] + 1):
            d[:, side, m] = sum(a[i] * (-k[i] ** 2) ** m * math.cos(k[i] * side + p[i]) * np.cos(k[i] * t)
                                for i in range(4))
    x = _coords(c["nx"], 1.0, "dirichlet")
    u0 = sum(float(a[i]) * torch.cos(float(k[i]) * x + float(p[i])) for i in range(4))
    return u0, d


def _source_data(c, seed):
    """The discrete delta at an interior node and a sinusoid turned on smoothly."""
    rng = np.random.default_rng(seed)
    ny, nx = _shape(c)
    hx, hy = 2.0 / (nx - 1), 2.0 / (ny - 1)
    g = torch.zeros(ny, nx, dtype=torch.float64, device=DEVICE)
    g[int(rng.integers(ny // 4, 3 * ny // 4)), int(rng.integers(nx // 4, 3 * nx // 4))] = 1.0 / (hx * hy)
    t = _dt(c) * np.arange(c["steps"] + 1)
    f = np.sin(rng.uniform(3.0, 5.0) * math.pi * t) * (1.0 - np.exp(-((t / 0.2) ** 2)))
    return torch.zeros_like(g), g, f


def _batch_problems(c):
    """Sizes, orders and CFL numbers of a batch: part of the case, the same for every seed."""
    rng = np.random.default_rng(c["count"] * 7919 + c["nmin"] + c["nmax"])
    n = np.exp(rng.uniform(math.log(c["nmin"]), math.log(c["nmax"]), size=c["count"])).round().astype(int)
    return ([(int(v), int(v)) for v in n], [int(v) for v in rng.integers(1, 4, size=c["count"])],
            [float(v) for v in rng.uniform(0.5, 4.0, size=c["count"])])


def _inputs(c, seed):
    """The inputs of a case as a dict of tensors and arrays, from the seed alone."""
    rng = np.random.default_rng(seed)
    if c["kind"] == "ends":
        u0, d = _end_data(c, seed)
        return {"u0": u0, "data": d}
    if c["kind"] == "source":
        u0, g, f = _source_data(c, seed)
        return {"u0": u0, "g": g, "f": f}
    if c["kind"] == "batch":
        shapes, _, _ = _batch_problems(c)
        return {"u0": torch.cat([_gaussian(s, rng, c["width"]).reshape(-1) for s in shapes])}
    if c["kind"] == "embedded":
        g = workloads.ellipse_grid(c["nx"])
        x = torch.from_numpy(g.x0 + g.hx * np.arange(g.nx)).to(DEVICE)
        cx, cy = rng.uniform(-0.3, 0.3, size=2)
        ex, ey = (torch.exp(-((x - m) ** 2) / (2 * c["width"] ** 2)) for m in (cx, cy))
        return {"geom": g, "u0": torch.where(torch.from_numpy(g.mask).to(DEVICE), ey[:, None] * ex[None, :], 0.0)}
    if c["kind"] == "plane" and c["bc"] == "dirichlet" or c["kind"] == "gradient":
        u0 = _gaussian(_shape(c), rng, c["width"])
    else:
        u0 = _modes(_shape(c), _length(c), c["bc"], rng, 8 if c["kind"] == "line" else 16,
                    8 if c["kind"] == "line" else 12)
    got = {"u0": u0}
    if c["kind"] == "gradient":
        ny, nx = _shape(c)
        flat = rng.choice((ny - 2) * (nx - 2), size=c["receivers"], replace=False)
        got["rec"] = np.sort((flat // (nx - 2) + 1) * nx + flat % (nx - 2) + 1).astype(np.int64)
        got["target"] = torch.from_numpy(0.1 * rng.normal(size=(c["steps"], c["receivers"]))).to(DEVICE)
    return got


# --------------------------------------------------------------------------
# One pass
# --------------------------------------------------------------------------
def prepare(case, seed):
    c = case
    s = dict(_inputs(c, seed), case=c)
    if c["kind"] == "batch":
        shapes, Ps, cfls = _batch_problems(c)
        s["solver"] = molt.BatchSolver(shapes, [f / (n - 1) for f, (n, _) in zip(cfls, shapes)], Ps, prec=c["prec"])
    elif c["kind"] == "embedded":
        s["solver"] = molt.EmbedSolver(s["geom"], dt=c["cfl"] * s["geom"].hx, P=c["P"], prec=c["prec"])
    else:
        shape, L = _shape(c), _length(c)
        lo = -1.0 if c["kind"] == "source" else 0.0
        s["solver"] = molt.Solver(shape, dt=_dt(c), P=c["P"], bc=c["bc"], prec=c["prec"], lo=[lo] * len(shape),
                                  hi=[lo + L] * len(shape))
    if c["kind"] == "gradient":
        s["u0"].requires_grad_(True)
    return s


def run(state):
    c, solver, u0 = state["case"], state["solver"], state["u0"]
    if c["kind"] == "ends":
        return solver.solve_dirichlet(u0, c["steps"], state["data"])
    if c["kind"] == "source":
        return solver.solve_source(u0, c["steps"], state["g"], state["f"])
    if c["kind"] == "gradient":
        t = molt.receiver_traces(u0, solver, state["rec"], c["steps"])
        grad, = torch.autograd.grad(t, u0, t.detach() - state["target"])
        return [t.detach(), grad]
    prev = u0.clone()
    cur = solver.start(prev)
    solver.step(prev, cur, c["steps"])
    return [prev, cur]


# --------------------------------------------------------------------------
# What a pass cannot do without
# --------------------------------------------------------------------------
def work(case):
    """A step reads two levels and writes one, 8 bytes a point each; a 1D line
    is read and written once per run.  A sweep of D along an axis costs 9
    operations a point (second difference 3, two recurrences 4, combination 2)."""
    c = case
    P, steps = c["P"], c["steps"] + (0 if c["kind"] in ("ends", "source", "gradient") else 1)
    if c["kind"] == "batch":
        shapes, Ps, _ = _batch_problems(c)
        pts = sum(a * b for a, b in shapes)
        sweeps = sum(a * b * 2 * p for (a, b), p in zip(shapes, Ps)) / pts
    elif c["kind"] == "embedded":
        pts, sweeps = int(workloads.ellipse_grid(c["nx"]).mask.sum()), 3 + 6 * (P - 1)
    else:
        pts = int(np.prod(_shape(c)))
        sweeps = {1: P, 2: 2 * P, 3: P * (P + 3)}[len(_shape(c))]
    if c["kind"] == "gradient":
        steps *= 2
    flops = steps * pts * (9.0 * sweeps + 4)
    if c["kind"] in ("line", "ends"):
        return {"bytes": 24.0 * pts, "flops": flops}
    return {"bytes": 24.0 * pts * steps, "flops": flops}


# --------------------------------------------------------------------------
# The method in float64 torch
# --------------------------------------------------------------------------
def _moment(k, nu):
    """int_0^nu t^k e^{-t} dt for an array nu, by its series where the closed form cancels."""
    nu = np.asarray(nu, dtype=np.float64)
    small = np.minimum(nu, 1.0)
    s, term = np.zeros_like(nu), small ** (k + 1)
    for i in range(40):
        s = s + term / (k + i + 1)
        term = term * (-small / (i + 1))
    e = np.exp(-nu)
    closed = [1 - e, 1 - (1 + nu) * e, 2 - (2 + 2 * nu + nu * nu) * e][k]
    return np.where(nu < 1.0, s, closed)


def _c(p, m, beta):
    return (-1) ** m * 2 * beta ** (2 * m) / math.factorial(2 * m) * math.comb(p - 1, m - 1)


def _beta_max(P):
    f = lambda b: -sum(_c(p, m, b) for p in range(1, P + 1) for m in range(1, p + 1)) - 4.0  # noqa: E731
    lo = 0.5
    while f(lo + 0.01) < 0:
        lo += 0.01
    hi = lo + 0.01
    for _ in range(100):
        mid = 0.5 * (lo + hi)
        lo, hi = (mid, hi) if f(mid) < 0 else (lo, mid)
    return 0.5 * (lo + hi)


def _causal(q, d):
    """y_j = d y_{j-1} + q_j along the last axis, y_{-1} = 0, by doubling."""
    s, g = 1, d
    while s < q.shape[-1] and g > 1e-25:
        q = torch.cat([q[..., :s], q[..., s:] + g * q[..., :-s]], dim=-1)
        s, g = 2 * s, g * g
    return q


def _anticausal(q, d):
    return _causal(q.flip(-1), d).flip(-1)


def _linv(v, nu, bc, ends=(0.0, 0.0)):
    """L^{-1} along the last axis of v (w = v - ends at Dirichlet ends)."""
    n, d = v.shape[-1], math.exp(-nu)
    m0, m1, m2 = (float(_moment(k, nu)) for k in (0, 1, 2))
    w0, w1, r = m0 - m1 / nu, m1 / nu, 0.5 * (m2 / nu ** 2 - m1 / nu)
    powers = torch.exp(-nu * torch.arange(n, dtype=torch.float64, device=v.device))
    if bc == "periodic":
        left, right = v.roll(1, -1), v.roll(-1, -1)
        S = right - 2 * v + left
        jl, jr = 0.5 * (w0 * v + w1 * left + r * S), 0.5 * (w0 * v + w1 * right + r * S)
        mu = math.exp(-nu * n)
        il, ir = _causal(jl, d), _anticausal(jr, d)
        # every periodic image: the full period's sum decays on around the ring
        il = il + il[..., -1:] / (1 - mu) * d * powers
        ir = ir + ir[..., :1] / (1 - mu) * d * powers.flip(-1)
        return il + ir
    S = v[..., 2:] - 2 * v[..., 1:-1] + v[..., :-2]
    sl, sr = torch.cat([S, S[..., -1:]], -1), torch.cat([S[..., :1], S], -1)
    zero = torch.zeros_like(v[..., :1])
    jl = torch.cat([zero, 0.5 * (w0 * v[..., 1:] + w1 * v[..., :-1] + r * sl)], -1)
    jr = torch.cat([0.5 * (w0 * v[..., :-1] + w1 * v[..., 1:] + r * sr), zero], -1)
    il, ir = _causal(jl, d), _anticausal(jr, d)
    mu = math.exp(-nu * (n - 1))
    r0 = v[..., :1] - ends[0] - ir[..., :1]
    r1 = v[..., -1:] - ends[1] - il[..., -1:]
    return il + ir + ((r0 - mu * r1) * powers + (r1 - mu * r0) * powers.flip(-1)) / (1 - mu * mu)


class _Box:
    """L^{-1} per axis on a rectangular grid; nu per array axis."""

    def __init__(self, shape, nu, bc):
        self.nd, self.nu, self.bc = len(shape), nu, bc

    def linv(self, v, a):
        return _linv(v.movedim(a, -1), self.nu[a], self.bc).movedim(-1, a)


class _Domain:
    """L^{-1} per axis on the line objects of an embedded domain."""

    def __init__(self, g, alpha):
        self.nd = 2
        self.ax = [self._lines(g.c0, g.c1, g.ca, g.cb, g.hy, alpha, g.ny),
                   self._lines(g.r0, g.r1, g.ra, g.rb, g.hx, alpha, g.nx)]

    @staticmethod
    def _weights(ts, length, alpha):
        """(alpha/2) int_0^length e^{-alpha s} l_i(s) ds of the Lagrange basis on the nodes ts."""
        m = [_moment(k, alpha * length) / alpha ** (k + 1) for k in range(3)]
        out = []
        for i in range(3):
            a, b = ts[(i + 1) % 3], ts[(i + 2) % 3]
            out.append(0.5 * alpha * (m[2] - (a + b) * m[1] + a * b * m[0]) / ((ts[i] - a) * (ts[i] - b)))
        return out

    def _lines(self, first, last, ga, gb, h, alpha, across):
        keep = np.nonzero(last >= first)[0]
        m = (last - first + 1)[keep]
        ga, gb = ga[keep], gb[keep]
        width, L = int(m.max()) + 2, len(keep)
        # node positions, column 0 = the first boundary point, column m + 1 = the second
        x = ga[:, None] + h * (np.arange(width)[None, :] - 1.0)
        x[:, 0] = 0.0
        x[np.arange(L), m + 1] = ga + (m - 1) * h + gb
        # past the line: any rising positions (never used)
        beyond = np.arange(width)[None, :] > (m + 1)[:, None]
        x = np.where(beyond, x[np.arange(L), m + 1][:, None] + h * (np.arange(width)[None, :] - (m + 1)[:, None]), x)
        wl, wr = np.zeros((3, L, width)), np.zeros((3, L, width))
        for dest, w, side in ((1, wl, -1), (0, wr, 1)):
            j = np.arange(dest, width if dest else width - 1)
            c0 = np.clip(np.broadcast_to(j - 1, (L, len(j))), 0, (m - 1)[:, None])
            ts = [side * (np.take_along_axis(x, np.minimum(c0 + i, width - 1), 1) - x[:, j]) for i in range(3)]
            w[:, :, j] = _Domain._weights(ts, side * (x[:, j + side] - x[:, j]), alpha)
        idx = first[keep][:, None] + np.arange(width)[None, :] - 1
        valid = (np.arange(width)[None, :] >= 1) & (np.arange(width)[None, :] <= m[:, None])
        dev = lambda t: torch.from_numpy(np.ascontiguousarray(t)).to(DEVICE)  # noqa: E731
        inside = (np.arange(width)[None, :] >= 1) & (np.arange(width)[None, :] <= (m + 1)[:, None])
        end = x[np.arange(L), m + 1]
        return {"keep": dev(keep), "idx": dev(np.clip(idx, 0, across - 1)), "valid": dev(valid),
                "wl": [dev(np.where(inside, t, 0.0)) for t in wl],
                "wr": [dev(np.where(valid | (np.arange(width)[None, :] == 0), t, 0.0)) for t in wr],
                "c0l": dev(np.clip(np.arange(width)[None, :] - 1, 0, (m - 1)[:, None])),
                "m": dev(m), "d": math.exp(-alpha * h), "mu": dev(np.exp(-alpha * end)),
                "ga": dev(np.exp(-alpha * ga)), "gb": dev(np.exp(-alpha * gb)), "ea": dev(np.exp(-alpha * x)),
                "eb": dev(np.exp(-alpha * np.maximum(end[:, None] - x, 0.0)))}

    def linv(self, v, a):
        t = self.ax[a]
        rows = v.movedim(a, -1)[t["keep"]]
        u = torch.where(t["valid"], rows.gather(1, t["idx"]), 0.0)
        width = u.shape[1]
        near = [u.gather(1, (t["c0l"] + i).clamp(max=width - 1)) for i in range(3)]
        jl = sum(w * n for w, n in zip(t["wl"], near))
        jr = sum(w * n for w, n in zip(t["wr"], near))
        last = t["m"][:, None] + 1
        # interior nodes decay by d per cell; the end cells by their own lengths
        il = _causal(torch.where(t["valid"], jl, 0.0), t["d"])
        il = torch.where(t["valid"], il, 0.0)
        ir = torch.where(t["valid"], _anticausal(torch.where(t["valid"], jr, 0.0), t["d"]), 0.0)
        il_b = t["gb"] * il.gather(1, t["m"][:, None])[:, 0] + jl.gather(1, last)[:, 0]
        ir_a = t["ga"] * ir[:, 1] + jr[:, 0]
        mu = t["mu"]
        A = (-ir_a + mu * il_b) / (1 - mu * mu)
        B = (-il_b + mu * ir_a) / (1 - mu * mu)
        w = torch.where(t["valid"], il + ir + A[:, None] * t["ea"] + B[:, None] * t["eb"], 0.0)
        back = torch.zeros_like(rows).scatter_add(1, t["idx"], w)
        out = torch.zeros_like(v.movedim(a, -1)).index_copy(0, t["keep"], back)
        return out.movedim(-1, a)


def _C(op, v):
    """sum over the axes of (prod of the other axes' L^{-1}) D v; x first."""
    axes = list(range(op.nd - 1, -1, -1))
    if op.nd == 1:
        return v - op.linv(v, 0)
    total = 0
    for a in axes:
        w = v - op.linv(v, a)
        for b in axes:
            if b != a:
                w = op.linv(w, b)
        total = total + w
    return total


def _D(op, v):
    w = v
    for a in range(op.nd):               # the outermost array axis first, x last
        w = op.linv(w, a)
    return v - w


def _F(op, u, P, beta):
    """sum_p sum_m c_pm C^m D^{p-m} u, built stage by stage in the order of
    Table 3: v[k] = C^{p-k} D^k u, the last one as D of the stage before it."""
    v, total = [], 0
    for p in range(1, P + 1):
        v = [_C(op, u)] if p == 1 else [_C(op, w) for w in v] + [_D(op, v[-1])]
        for k, w in enumerate(v):
            total = total + _c(p, p - k, beta) * w
    return total


def _march(op, u0, steps, P, beta):
    prev, cur = u0, u0 + 0.5 * _F(op, u0, P, beta)
    for _ in range(steps):
        prev, cur = cur, 2 * cur - prev + _F(op, cur, P, beta)
    return prev, cur


def _transposed(op, w, P, beta):
    x = torch.zeros_like(w, requires_grad=True)
    with torch.enable_grad():
        return torch.autograd.grad(_F(op, x, P, beta), x, w)[0]


def _nus(c, beta):
    alpha = beta / _dt(c)
    return alpha, [alpha * _spacing(n, _length(c), c["bc"]) for n in _shape(c)]


def exact(case, seed):
    c = case
    s = _inputs(c, seed)
    u0, P, steps = s["u0"], c["P"], c["steps"]
    if c["kind"] == "batch":
        shapes, Ps, cfls = _batch_problems(c)
        prev, cur, at = [], [], 0
        for shape, p, cfl in zip(shapes, Ps, cfls):
            b = _beta_max(p)
            a0 = u0[at:at + shape[0] * shape[1]].view(shape)
            at += shape[0] * shape[1]
            for to, v in zip((prev, cur), _march(_Box(shape, [b / cfl] * 2, "dirichlet"), a0, steps, p, b)):
                to.append(v.reshape(-1))
        return [torch.cat(prev), torch.cat(cur)]
    beta = _beta_max(P)
    if c["kind"] == "embedded":
        return list(_march(_Domain(s["geom"], beta / (c["cfl"] * s["geom"].hx)), u0, steps, P, beta))
    alpha, nu = _nus(c, beta)
    if c["kind"] == "ends":
        gam = s["data"] / alpha ** (2 * np.arange(P + 1))
        prev, cur = None, u0
        for k in range(steps):
            v, F = cur, 0
            for p in range(1, P + 1):
                ends = [(-1) ** p * sum(math.comb(j - 1, p - 1) * float(gam[k, side, j]) for j in range(p, P + 1))
                        for side in (0, 1)]
                v = v - _linv(v, nu[0], "dirichlet", ends)
                F = F + sum(_c(p, m, beta) for m in range(1, p + 1)) * v
            new = cur + 0.5 * F if k == 0 else 2 * cur - prev + F
            new = torch.cat([new.new_tensor([s["data"][k + 1, 0, 0]]), new[1:-1],
                             new.new_tensor([s["data"][k + 1, 1, 0]])])
            prev, cur = cur, new
        return cur
    op = _Box(_shape(c), nu, c["bc"])
    if c["kind"] == "source":
        g, f, sc = s["g"], s["f"], _dt(c) ** 2
        Cg = _C(op, g)
        prev, cur = None, u0
        for k in range(steps):
            before = f[k - 1] if k else f[1]
            a, b = (sc * f[k], 0.0) if P == 1 else (sc * (f[k + 1] + 10 * f[k] + before) / 12,
                                                    -beta ** 2 * sc * f[k] / 12)
            push = _F(op, cur, P, beta) + float(a) * g + float(b) * Cg
            prev, cur = cur, cur + 0.5 * push if k == 0 else 2 * cur - prev + push
        return cur
    if c["kind"] == "gradient":
        rec = torch.from_numpy(s["rec"]).to(DEVICE)
        prev, cur, t = u0, u0 + 0.5 * _F(op, u0, P, beta), []
        for _ in range(steps):
            t.append(cur.reshape(-1)[rec])
            prev, cur = cur, 2 * cur - prev + _F(op, cur, P, beta)
        t = torch.stack(t)
        w = t - s["target"]
        mu, later = torch.zeros_like(u0), torch.zeros_like(u0)
        for n in range(steps, 0, -1):
            new = 2 * mu - later + _transposed(op, mu, P, beta)
            new.view(-1).index_add_(0, rec, w[n - 1])
            mu, later = new, mu
        return [t, mu + 0.5 * _transposed(op, mu, P, beta) - later]
    return list(_march(op, u0, steps, P, beta))
