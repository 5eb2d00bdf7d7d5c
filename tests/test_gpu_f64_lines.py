"""The float64 line passes against the oracle at the sizes where they can go
wrong: lines shorter than a segment, segment edges and remainders, a last
segment of one point, decays whose inflow window covers the line (and exceeds
it), the longest lines the passes take and the first that fall back, rows that
start off a 32-byte boundary.

Tolerance: 1e-12 relative L2, or 64 eps64 |v| / |D v| where the oracle's own
subtraction v - L^{-1} v loses more (as in test_gpu_parity).
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle
from test_gpu_parity import cond_of, dev, field, make, rel_l2, spacing, tol_for

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [3, 4, 7, 8, 9, 10, 15, 16, 17, 31, 32, 33, 63, 65, 127, 129, 255, 257, 1025])
@pytest.mark.parametrize("bc", ["dirichlet", "periodic"])
@pytest.mark.parametrize("cfl", [0.3, 2.0, 60.0])
def test_powers_on_both_axes_match_oracle(n, bc, cfl):
    m = 5
    for shape, axis in (((n, m), 1), ((m, n), 0)):
        for quad in (2, 1):
            s = make(shape, cfl * spacing(n, bc), 2, bc, "fp64", quad)
            v = field(shape, 200 + n, bc)
            for power in (1, 3):
                got = s.apply_D(dev(v), axis, power).cpu().numpy()
                ref = oracle.D_axis(v, axis, s.nu[axis], bc, quad, power=power)
                err = rel_l2(got, ref)
                assert err <= tol_for("fp64", s, power, cond_of(v, ref)), (shape, axis, quad, power, err)
            s.close()


@pytest.mark.parametrize("shape, axis", [((3, 8192), 0), ((3, 8193), 0), ((4096, 3), 1), ((4097, 3), 1)])
def test_longest_lines_and_their_fallback_match_oracle(shape, axis):
    n, bc = max(shape), "dirichlet"
    s = make(shape, 2.0 * spacing(n, bc), 2, bc, "fp64")
    v = field(shape, 210, bc)
    got = s.apply_D(dev(v), axis, 2).cpu().numpy()
    ref = oracle.D_axis(v, axis, s.nu[axis], bc, 2, power=2)
    assert rel_l2(got, ref) <= tol_for("fp64", s, 2, cond_of(v, ref))
    u = dev(v)
    F = s.apply_F(u).cpu().numpy()
    rF = oracle.F(v, s.nu, 2, s.beta, bc)
    assert rel_l2(F, rF) <= tol_for("fp64", s, 4, cond_of(v, rF))
    s.close()


@pytest.mark.parametrize("shape, P", [((3, 3), 5), ((17, 9), 3), ((33, 31), 3), ((100, 96), 2), ((9, 11, 13), 3),
                                      ((40, 33, 8), 2), ((75, 100, 96), 1)])
@pytest.mark.parametrize("bc", ["dirichlet", "periodic"])
def test_operator_and_steps_match_oracle(shape, P, bc):
    s = make(shape, 1.5 * spacing(min(shape), bc), P, bc, "fp64")
    u = field(shape, 220, bc)
    F = s.apply_F(dev(u)).cpu().numpy()
    ref = oracle.F(u, s.nu, P, s.beta, bc)
    assert rel_l2(F, ref) <= tol_for("fp64", s, 2 * P, cond_of(u, ref))
    u1 = s.start(dev(u))
    up, uc = dev(u), u1.clone()
    s.step(up, uc, 5)
    rp, rc = oracle.run(u, oracle.start(u, s.nu, P, s.beta, bc), 5, s.nu, P, s.beta, bc)
    assert rel_l2(up.cpu().numpy(), rp) <= 1e-12 and rel_l2(uc.cpu().numpy(), rc) <= 1e-12
    s.close()


@pytest.mark.parametrize("nx", [256, 100, 37])
def test_fields_off_a_vector_boundary_give_the_same_bits(nx):
    """Rows that start on 32 bytes are read in vectors, others point by point."""
    shape = (24, nx)
    s = make(shape, 0.01, 3, "dirichlet", "fp64")
    u = dev(field(shape, 230, "dirichlet"))
    want = s.apply_F(u)
    for off in (1, 2):
        buf = torch.zeros(u.numel() + 4, dtype=torch.float64, device="cuda")
        out = torch.zeros_like(buf)
        us, os_ = buf[off:off + u.numel()].view(shape), out[off:off + u.numel()].view(shape)
        us.copy_(u)
        s.apply_F(us, out=os_)
        assert torch.equal(os_, want)
        assert not out[:off].any() and not out[off + u.numel():].any()
    s.close()
