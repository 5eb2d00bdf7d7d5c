"""The float64 passes at both ends of the decay per cell, nu = alpha h.

Very slow decay (a domain far shorter than 1 / alpha): every segment sees every
other one.  On a field that vanishes at both ends L^{-1} v is below (nu + (n nu)^2)
|v| (the quadratic rule's own term and the domain's length), so D v is v
itself.  Tolerance: that, plus 2 n eps64 / nu for the solve, which sums n values
rounded once (second differences, at most 4 |v|) with the response 1 / (2 nu) of
the open line and takes the two end terms out again.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle
from paper_1308_3214_gb300 import workloads
from test_gpu_parity import cond_of, dev, field, make, rel_l2, spacing, tol_for

pytestmark = pytest.mark.gpu

EPS64 = 2.0 ** -52


def slow_tol(n, nu):
    return 2 * n * EPS64 / nu + nu + (n * nu) ** 2


# nu times 4 points a segment below 60 ln 2 / 2^31: the number of segments whose
# inflow matters exceeds an int.  Lines whose last segment is full and short.
SLOW = [1e-9, 4e-9, 3e-11]


@pytest.mark.parametrize("n", [5, 64, 301, 1000])
@pytest.mark.parametrize("nu", SLOW)
@pytest.mark.parametrize("quad", [1, 2])
def test_powers_of_slow_decay(n, nu, quad):
    for shape, axis in (((n, 3), 1), ((3, n), 0)):
        s = make(shape, oracle.beta_max(2) * spacing(n, "dirichlet") / nu, 2, "dirichlet", "fp64", quad)
        assert abs(s.nu[axis] / nu - 1) < 1e-12
        v = np.zeros(shape)
        line = field((n,), 400 + n, "dirichlet")
        line[0] = line[-1] = 0.0
        v[:] = line[:, None] if axis == 1 else line[None, :]
        got = s.apply_D(dev(v), axis, 1).cpu().numpy()
        assert rel_l2(got, v) <= slow_tol(n, nu), (shape, rel_l2(got, v))
        s.close()


@pytest.mark.parametrize("n", [5, 64, 301, 1000, 3001])
@pytest.mark.parametrize("nu", SLOW)
def test_line_loop_of_slow_decay(n, nu):
    """One step of the 1D loop against the level update with F[u] = f_1 D u = -beta^2 u
    (P = 1)."""
    beta = oracle.beta_max(1)
    s = make((n,), beta * spacing(n, "dirichlet") / nu, 1, "dirichlet", "fp64")
    u0, u1 = (field((n,), 410 + k, "dirichlet") for k in (0, 1))
    u0[0] = u0[-1] = u1[0] = u1[-1] = 0.0
    up, uc = dev(u0), dev(u1)
    s.step(up, uc, 1)
    ref = 2 * u1 - u0 - beta ** 2 * u1
    assert np.array_equal(up.cpu().numpy(), u1)
    assert rel_l2(uc.cpu().numpy(), ref) <= beta ** 2 * slow_tol(n, nu) * np.linalg.norm(u1) / np.linalg.norm(ref)
    s.close()


@pytest.mark.parametrize("nu", SLOW)
def test_batch_of_slow_decay(nu):
    """Two ragged problems, P = 1: F u = -beta^2 (D_x + D_y - 2 D_x D_y) u, nothing but
    the errors of four applications where D is the identity."""
    from paper_1308_3214_gb300 import molt
    beta = oracle.beta_max(1)
    ns = (61, 130)
    b = molt.BatchSolver([(n, n) for n in ns], dt=[beta * spacing(n, "dirichlet") / nu for n in ns], P=1, prec="fp64")
    us = [field((n, n), 420 + n, "dirichlet") for n in ns]
    got = b.apply_F(dev(np.concatenate([u.ravel() for u in us]))).cpu().numpy()
    o = 0
    for n, u in zip(ns, us):
        F = got[o:o + n * n]
        o += n * n
        assert np.linalg.norm(F) <= 4 * beta ** 2 * slow_tol(n, nu) * np.linalg.norm(u), n
    b.close()


@pytest.mark.parametrize("n", [24, 260])
@pytest.mark.parametrize("nu", SLOW)
@pytest.mark.parametrize("axis", [0, 1])
def test_embedded_lines_of_slow_decay(n, nu, axis):
    """L^{-1} v = v - D v vanishes on a disk far smaller than 1 / alpha (the rounding of an
    end cell's second difference grows with the spacing over the shortest gap)."""
    from paper_1308_3214_gb300 import molt
    g = workloads.disk_grid(n)
    live = g.mask.any(axis=1 - axis)
    gaps = (g.ra[live], g.rb[live]) if axis == 0 else (g.ca[live], g.cb[live])
    gmin = min(x.min() for x in gaps)
    s = molt.EmbedSolver(g, dt=oracle.beta_max(1) * g.hx / nu, P=1)
    v = workloads.random_field((n, n), 430 + n) * g.mask
    w = s.linv(dev(v), axis).cpu().numpy()
    assert np.linalg.norm(w) <= slow_tol(n, nu) * (g.hx / gmin) * np.linalg.norm(v)
    s.close()


# ---------------------------------------------------------------------------
# Very fast decay: below d = 1e-140 (nu = 322.4) nothing divides by d any more.
# The end nodes of an embedded line stand gaps of any length away from the
# boundary points, so the terms of the two ends still reach them.
# Tolerances: as in test_gpu_embedded, 100 eps64 over the shortest gap in cells;
# mixed: 16 roundings of the decay sum, 2 eps32 each, of the field.
# ---------------------------------------------------------------------------
FAST = [80.0, 321.0, 323.0, 400.0, 1000.0]


def notched_grid(gaps):
    """A rectangle of 9 x 7 interior nodes with a column of two more above it (rows of
    one node) and a row of three more beside it; the gaps are dealt out in turn,
    in spacings."""
    ny, nx, h = 12, 15, 0.1
    mask = np.zeros((ny, nx), bool)
    mask[1:8, 2:11] = True
    mask[8:10, 5] = True
    mask[3, 11:14] = True
    k = [0]

    def line(m):
        n = len(m)
        lo, hi = np.ones(n, np.int64), np.zeros(n, np.int64)
        ga, gb = np.zeros(n), np.zeros(n)
        for i in range(n):
            j = np.flatnonzero(m[i])
            if len(j) == 0:
                continue
            lo[i], hi[i] = j[0], j[-1]
            ga[i], gb[i] = (h * gaps[(k[0] + q) % len(gaps)] for q in (0, 1))
            k[0] += 1
        return lo, hi, ga, gb
    r0, r1, ra, rb = line(mask)
    c0, c1, ca, cb = line(mask.T)
    return workloads.EmbeddedGrid(nx, ny, 0.0, 0.0, h, h, r0, r1, ra, rb, c0, c1, ca, cb, mask)


@pytest.mark.parametrize("nu", FAST)
@pytest.mark.parametrize("gaps", [(1e-6, 0.7), (1e-3, 1e-6, 1.0), (1e-6,)])
def test_embedded_lines_of_fast_decay(nu, gaps):
    from paper_1308_3214_gb300 import molt
    g = notched_grid(gaps)
    P, beta, alpha = 2, oracle.beta_max(2), nu / g.hx
    s = molt.EmbedSolver(g, dt=beta / alpha, P=P)
    v = workloads.random_field((g.ny, g.nx), 440) * g.mask
    tol = 100 * EPS64 / min(gaps)
    for axis in (0, 1):
        got = s.linv(dev(v), axis).cpu().numpy()
        ref = oracle.linv_axis_embed(v, axis, g, alpha)
        assert rel_l2(got, ref) <= tol, (axis, rel_l2(got, ref))
    assert rel_l2(s.apply_F(dev(v)).cpu().numpy(), oracle.F_embed(v, g, alpha, P, beta)) <= tol
    s.close()


# float32 sweeps: e^{alpha h} exceeds a float at nu = 88.7, d is zero at 104
@pytest.mark.parametrize("nu", [79.0, 81.0, 88.5, 89.0, 95.0, 110.0, 323.0, 1000.0])
@pytest.mark.parametrize("gaps", [(0.5, 0.9), (1e-3, 0.7), (1e-3, 1e-2, 1.0), (2.5, 1e-3)])
def test_mixed_embedded_lines_of_fast_decay(nu, gaps):
    """Bounds of test_gpu_embedded: 16 eps32 (1 + 1 / (1 - d)), of the field for L^{-1} v, times
    2P of F."""
    from paper_1308_3214_gb300 import molt
    g = notched_grid(gaps)
    P, beta, alpha = 2, oracle.beta_max(2), nu / g.hx
    s = molt.EmbedSolver(g, dt=beta / alpha, P=P, prec="mixed")
    v = workloads.random_field((g.ny, g.nx), 441) * g.mask
    tol = 16 * 2 * 2.0 ** -24 + 100 * EPS64 / min(gaps)
    for axis in (0, 1):
        got = s.linv(dev(v), axis).cpu().numpy()
        ref = oracle.linv_axis_embed(v, axis, g, alpha)
        assert np.linalg.norm(got - ref) <= tol * np.linalg.norm(v), axis
    F = oracle.F_embed(v, g, alpha, P, beta)
    assert rel_l2(s.apply_F(dev(v)).cpu().numpy(), F) <= 2 * P * tol
    s.close()


@pytest.mark.parametrize("nu", [740.0, 746.0, 1200.0])
@pytest.mark.parametrize("shape", [(77, 4), (5, 130), (33, 31)])
@pytest.mark.parametrize("prec", ["fp64", "mixed"])
def test_batches_of_a_decay_below_the_float64_range(nu, shape, prec):
    """d = e^{-nu} is zero from nu = 745.2 on (a few points across a long axis, or a tiny
    step): F and F^T of batches and of ragged handles."""
    from paper_1308_3214_gb300 import molt
    P, beta = 2, oracle.beta_max(2)
    dt = beta * spacing(min(shape), "dirichlet") / nu
    s = make(shape, dt, P, "dirichlet", prec)
    b = molt.BatchSolver([shape, shape], dt=dt, P=P, prec=prec)
    v = field(shape, 450, "dirichlet")
    for one, many, ref in ((s.apply_F, b.apply_F, oracle.F), (s.apply_FT, b.apply_FT, oracle.FT)):
        want = ref(v, s.nu, P, beta, "dirichlet")
        tol = tol_for(prec, s, 2 * P, cond_of(v, want))
        assert rel_l2(one(dev(v)).cpu().numpy(), want) <= tol
        got = many(dev(np.concatenate([v.ravel()] * 2))).cpu().numpy().reshape((2,) + shape)
        assert rel_l2(got[0], want) <= tol and np.array_equal(got[0], got[1])
    b.close()
    s.close()
