"""Segments per CTA of the float32 strided passes: what a handle reports and what
a caller sets is what runs, and the tensor stores of 5, 6 or 7 segments of 64
rows per CTA (no whole number of 256-row boxes) against the oracle.

A column of n points has G = n / 64 segments, over K = ceil(G / w) CTAs (w:
strided_warps) of ceil(G / K) each.
"""
import pytest

torch = pytest.importorskip("torch")

import oracle
from test_gpu_parity import dev, field, make, rel_l2, spacing, tol_for

pytestmark = pytest.mark.gpu


def segments_per_cta(n, warps):
    G = n // 64
    K = -(-G // warps)
    return -(-G // K)


# narrow grids whose columns run over clusters of 2 or more: fewer segments per
# CTA; columns that fit one CTA, and grids with a CTA for every SM: 8
@pytest.mark.parametrize("shape, warps", [((1024, 1024), {2, 4}), ((2048, 96), {4}), ((640, 640), {2}),
                                          ((256, 256), {8}), ((512, 512), {8}), ((448, 64), {8}),
                                          ((2048, 2048), {8}), ((896, 4896), {8})])
@pytest.mark.parametrize("bc", ["dirichlet", "periodic"])
def test_the_reported_split_runs_and_does_not_change_the_bits(shape, warps, bc):
    s = make(shape, 2.0 * spacing(max(shape), bc), 2, bc, "mixed")
    cur = s.tuning()
    assert cur["strided_warps"] in warps
    v = dev(field(shape, 95, bc))
    got = [s.apply_D(v, 1, p).clone() for p in (1, 2)]
    for w in (8, cur["strided_warps"]):
        s.set_tuning(cur["res_warps"], cur["strided_rpt"], w, cur["rows_warps"])
        assert s.tuning()["strided_warps"] == w
        for p in (1, 2):
            assert torch.equal(s.apply_D(v, 1, p), got[p - 1]), (w, p)
    s.close()


def test_a_slowly_decaying_column_keeps_its_split():
    """The full-carry passes (no neighbour exchange) run 8 segments per CTA unless told
    otherwise."""
    s = make((1024, 64), 60.0 * spacing(1024, "periodic"), 2, "periodic", "mixed")
    assert s.tuning()["strided_warps"] == 8
    s.close()


@pytest.mark.parametrize("shape, S", [((320, 36), 5), ((384, 100), 6), ((448, 4864), 7), ((640, 2432), 5),
                                      ((832, 2500), 7), ((896, 2432), 7)])
@pytest.mark.parametrize("bc", ["dirichlet", "periodic"])
@pytest.mark.parametrize("stage", [2, 3])
def test_default_tensor_stores_of_uneven_segment_counts(shape, S, bc, stage):
    ny = shape[0]
    s = make(shape, 1.5 * spacing(ny, bc), 3, bc, "mixed")
    cur = s.tuning()
    assert segments_per_cta(ny, cur["strided_warps"]) == S and cur["strided_stage"] == 2
    if stage != cur["strided_stage"]:
        s.set_tuning(cur["res_warps"], cur["strided_rpt"], cur["strided_warps"], cur["rows_warps"], strided_stage=stage)
    v = field(shape, 96, bc)
    vd = dev(v)
    for p in (1, 2, 3):
        got = s.apply_D(vd, 1, p).cpu().numpy()
        ref = oracle.D_axis(v, 1, s.nu[1], bc, 2, power=p)
        assert rel_l2(got, ref) <= tol_for("mixed", s, p), (p, rel_l2(got, ref))
    s.sync()
    s.close()
