"""F^T on ragged Dirichlet grids needs no memory of its own at the call: the first
call of a new handle can be captured in a CUDA graph, in both precisions, and
replayed on new values."""
import pytest

torch = pytest.importorskip("torch")

import oracle
from test_gpu_parity import dev, field, make, rel_l2, tol_for

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(77, 100), (130, 61)])
@pytest.mark.parametrize("prec", ["fp64", "mixed"])
def test_first_transposed_call_can_be_captured(shape, prec):
    s = make(shape, 0.02, 2, "dirichlet", prec)
    ws = [field(shape, 500 + k, "dirichlet") for k in range(2)]
    w, out = dev(ws[0]), torch.zeros(shape, dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        s.apply_FT(w, out=out)
    for v in ws:
        w.copy_(dev(v))
        g.replay()
        ref = oracle.FT(v, s.nu, 2, s.beta, "dirichlet")
        assert rel_l2(out.cpu().numpy(), ref) <= tol_for(prec, s, 4)
    s.close()
