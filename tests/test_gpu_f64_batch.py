"""The float64 passes of a batch, forward and transposed, against the oracle at
the sizes where they can go wrong: lines shorter than a segment, segment edges
and remainders, a last segment of one point (the point next to the end lies in
the segment before it), rows padded by 1, 2 and 3 points, the longest lines,
decays whose inflow window covers the line, both quadrature orders.

Tolerance: 1e-12 relative L2, or 64 eps64 |u| / |F u| where the oracle's own
subtraction v - L^{-1} v loses more (as in test_gpu_batch).
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle
from paper_1308_3214_gb300 import molt

pytestmark = pytest.mark.gpu

EPS64 = 2.0 ** -52
EDGES = [3, 4, 5, 6, 8, 9, 16, 17, 18, 31, 32, 33, 34, 65, 129, 255, 257, 513, 1023, 1024]
SHAPES = [(n, 7) for n in EDGES] + [(6, n) for n in EDGES] + [(3, 3), (33, 65), (97, 129), (257, 513)]


def rel_l2(a, b):
    den = np.linalg.norm(b)
    return np.linalg.norm(a - b) / (den if den > 0 else 1.0)


@pytest.mark.parametrize("cfl", [0.3, 2.0, 60.0])
@pytest.mark.parametrize("quad", [2, 1])
def test_F_and_its_transpose_match_oracle(cfl, quad):
    Ps = [1 + i % 5 for i in range(len(SHAPES))]
    dts = [cfl / (max(s) - 1) for s in SHAPES]
    b = molt.BatchSolver(SHAPES, dt=dts, P=Ps, prec="fp64", quad_order=quad)
    rng = np.random.default_rng(41)
    us = [rng.normal(size=s) for s in SHAPES]
    F, FT = b.unpack(b.apply_F(b.pack(us))), b.unpack(b.apply_FT(b.pack(us)))
    torch.cuda.synchronize()
    for i, (u, shape, P, dt) in enumerate(zip(us, SHAPES, Ps, dts)):
        beta = oracle.beta_max(P)
        nu = tuple(beta / dt / (n - 1) for n in (shape[1], shape[0]))
        for got, ref in ((F[i], oracle.F(u, nu, P, beta, "dirichlet", quad)),
                         (FT[i], oracle.FT(u, nu, P, beta, "dirichlet", quad))):
            cond = np.linalg.norm(u) / max(np.linalg.norm(ref), 1e-300)
            assert rel_l2(got.cpu().numpy(), ref) <= max(1e-12, 64 * EPS64 * cond), (shape, P)
    b.close()
