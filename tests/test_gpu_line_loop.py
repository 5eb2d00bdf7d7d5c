"""1D time loops run many steps per launch: the float32 forms against one
launch per step (use_graphs=False), bit for bit -- whole segments on one warp,
ragged lines on one warp and on a whole CTA, with and without boundary data --
and the float64 form against the oracle over splits into warps and CTAs, inflow
windows that cover the line, and runs longer than one launch's boundary data.

Float64 tolerance: 1e-12 relative L2, as test_gpu_parity, or 16 eps64 P / (1 -
d)^2 a step where the decay is so slow that this is more (the difference form
passes the rounding of a periodic line's mean on times 1 / (1 - d)^2); with boundary data
64 eps64 per step times the size of the end terms against the field where that
is more (both sides add A_p times the end values of D^p u, which on 3 points at
CFL 2 are 10^6 times the field).
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle
from test_gpu_parity import dev, field, make, rel_l2, smooth_field, spacing

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [3, 33, 64, 256, 500, 1000, 1023, 1024, 1500, 2048, 3001, 12288])
@pytest.mark.parametrize("bc", ["dirichlet", "periodic"])
@pytest.mark.parametrize("P", [1, 3])
def test_float32_loop_gives_the_bits_of_single_steps(n, bc, P):
    u0 = smooth_field((n,), 300, bc) + 0.01 * field((n,), 301, bc)
    for nsteps in (1, 6):
        outs = []
        for graphs in (True, False):
            s = make((n,), 1.5 * spacing(n, bc), P, bc, "mixed", use_graphs=graphs)
            up = dev(u0)
            uc = s.start(up)
            s.step(up, uc, nsteps)
            outs.append((up, uc))
            s.close()
        assert torch.equal(outs[0][0], outs[1][0]) and torch.equal(outs[0][1], outs[1][1])


def end_data(n, P, dt, nsteps):
    """cos(3 pi x) cos(3 pi t) + cos(x) cos(t) and its end data."""
    t = dt * np.arange(nsteps + 1)
    d = np.zeros((nsteps + 1, 2, P + 1))
    for k in (3 * np.pi, 1.0):
        for side in (0, 1):
            for m in range(P + 1):
                d[:, side, m] += (-k * k) ** m * np.cos(k * side) * np.cos(k * t)
    x = np.linspace(0.0, 1.0, n)
    return np.cos(3 * np.pi * x) + np.cos(x), d


@pytest.mark.parametrize("n", [3, 40, 200, 999, 1024, 3001, 10001])
@pytest.mark.parametrize("nsteps", [1, 50])
def test_float32_boundary_data_loop_gives_the_bits_of_single_steps(n, nsteps):
    dt = 2.0 * spacing(n, "dirichlet")
    u0, d = end_data(n, 3, dt, nsteps)
    outs = []
    for graphs in (True, False):
        s = make((n,), dt, 3, "dirichlet", "mixed", use_graphs=graphs)
        outs.append(s.solve_dirichlet(dev(u0), nsteps, d))
        s.close()
    assert torch.equal(outs[0], outs[1])


@pytest.mark.parametrize("n", [3, 4, 63, 64, 65, 129, 255, 256, 257, 1000, 2049, 3205, 8192, 12288])
@pytest.mark.parametrize("bc", ["dirichlet", "periodic"])
@pytest.mark.parametrize("cfl", [0.3, 1.5, 60.0])
def test_float64_loop_matches_oracle(n, bc, cfl):
    for P in (1, 3):
        s = make((n,), cfl * spacing(n, bc), P, bc, "fp64")
        u0 = smooth_field((n,), 310, bc) + 0.01 * field((n,), 311, bc)
        u1 = oracle.start(u0, s.nu, P, s.beta, bc)
        up, uc = dev(u0), dev(u1)
        s.step(up, uc, 7)
        rp, rc = oracle.run(u0, u1, 7, s.nu, P, s.beta, bc)
        tol = max(1e-12, 7 * 16 * 2.0 ** -52 * P / (1.0 - s.d[0]) ** 2)
        assert rel_l2(up.cpu().numpy(), rp) <= tol and rel_l2(uc.cpu().numpy(), rc) <= tol, P
        s.close()


@pytest.mark.parametrize("n", [3, 65, 200, 1025, 10001])
@pytest.mark.parametrize("nsteps", [1, 60])
def test_float64_boundary_data_loop_matches_oracle(n, nsteps):
    P, dt = 3, 2.0 * spacing(n, "dirichlet")
    u0, d = end_data(n, P, dt, nsteps)
    s = make((n,), dt, P, "dirichlet", "fp64")
    got = s.solve_dirichlet(dev(u0), nsteps, d).cpu().numpy()
    gam = d / s.alpha ** (2 * np.arange(P + 1))
    ref = oracle.run_bc(u0, nsteps, s.nu[0], P, s.beta, gam)
    ends = max(np.abs(oracle.Ap(P, s.beta)) @ np.abs(oracle.bc_values(g, P)[1:]).max(axis=1) for g in gam)
    tol = max(1e-12, 64 * 2.0 ** -52 * nsteps * ends / np.sqrt(np.mean(ref ** 2)))
    assert rel_l2(got, ref) <= tol
    s.close()
