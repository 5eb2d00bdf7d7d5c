"""F^T of the mixed batched passes on columns whose last segment holds one, two,
three points, at every segment length (4, 8, 16, 32, 64 points), and on rows of
the same lengths; bound of test_gpu_parity for 2P applications."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle
from test_gpu_parity import dev, field, make, rel_l2, spacing, tol_for

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [5, 6, 7, 10, 14, 17, 18, 19, 26, 33, 34, 35, 50, 65, 66, 67, 98, 129, 130, 131, 194, 258, 514,
                               770, 1010, 1022])
@pytest.mark.parametrize("cfl", [0.7, 2.5, 12.0])
def test_transpose_with_a_short_last_segment(n, cfl):
    for shape in ((n, 37), (37, n)):
        s = make(shape, cfl * spacing(n, "dirichlet"), 2, "dirichlet", "mixed")
        w = field(shape, 600 + n, "dirichlet")
        got = s.apply_FT(dev(w)).cpu().numpy()
        ref = oracle.FT(w, s.nu, 2, s.beta, "dirichlet")
        assert rel_l2(got, ref) <= tol_for("mixed", s, 4), (shape, rel_l2(got, ref))
        s.close()


def test_gradient_of_a_run_with_a_short_last_segment():
    """The trace gradient's inner product with a direction is the traces' with their
    gradient (a linear map and its transpose), to the mixed bound."""
    shape, nsteps = (130, 61), 12
    s = make(shape, 0.02, 2, "dirichlet", "mixed")
    rec = np.array([64 * 61 + 30, 127 * 61 + 20, 100 * 61 + 5])
    u = field(shape, 610, "dirichlet")
    tg = torch.from_numpy(np.random.default_rng(611).normal(size=(nsteps, rec.size))).cuda()
    tr = s.traces(dev(u), rec, nsteps)
    grad = s.adjoint(rec, tg)
    a, b = float((tr * tg).sum()), float((grad * dev(u)).sum())
    size = float(tr.norm() * tg.norm())
    assert abs(a - b) <= nsteps * tol_for("mixed", s, 4) * size
    s.close()
