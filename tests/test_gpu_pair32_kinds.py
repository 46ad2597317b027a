"""FP32 pair sums and treecode over the row pairs that have a loop of their own (V/K rows: the direct forms and both
kernels in a row; V/K + D/T rows: no Yukawa term, both kernels everywhere, and the rest), against the library's FP64
application, which the parity tests hold to the oracle. Tolerances as there and in the treecode's test: FP32 2e-5,
split-coordinate FP32 2e-6, treecode 1e-4."""
import pytest

from synth.icosphere import uv_ellipsoid

pytestmark = pytest.mark.gpu

# (form, alpha, beta); cfie_ext with alpha = 0 has a row without Laplace terms, cfie_int with alpha = beta = 0 no Yukawa
FORMS = [("direct_int", 0, 0), ("direct_ext_perm", 0, 0), ("juffer", 0, 0), ("lu", 0, 0), ("pmchwt_ext", 0, 0),
         ("cfie_ext", 0.0, 0.5), ("cfie_int", 0.0, 0.0), ("cfie_int", 0.7, 0.0)]


@pytest.mark.parametrize("form,alpha,beta", FORMS)
@pytest.mark.parametrize("n_lon,n_lat,far_q", [(13, 11, 6), (21, 24, 3)])  # 1,560 and 2,898 points
def test_row_kinds(form, alpha, beta, n_lon, n_lat, far_q):
    import torch

    import paper_2108_10481_gb300 as pb
    v, t = uv_ellipsoid(n_lon, n_lat, (2.0, 1.6, 1.3), center=(0.3, -0.2, 0.1), twist=0.1)
    ctx = pb.pb_init(0)
    m = pb.pb_mesh_load(ctx, v, t, far_q=far_q, n_ss=3)
    nf = pb.pb_near_build(ctx, m, 0.125)
    P = pb.Params(4.0, 80.0, 0.125)
    x = torch.randn(2 * v.shape[0], dtype=torch.float64, device="cuda", generator=torch.Generator("cuda").manual_seed(1))

    def apply(prec):
        return pb.pb_system_apply(ctx, m, nf, P, form, x, prec=prec, alpha=alpha, beta=beta)

    ref = apply(pb.PB_F64)
    for prec, tree, tol in ((pb.PB_F32, False, 2e-5), (pb.PB_F32_ACCURATE, False, 2e-6), (pb.PB_F32, True, 1e-4)):
        pb.pb_set_treecode(ctx, tree, 6, 0.7, 0)
        y = apply(prec)
        assert float((y - ref).norm() / ref.norm()) < tol, (prec, tree)


@pytest.mark.parametrize("form,alpha,beta", FORMS)
def test_centroid_rule(form, alpha, beta):
    """One point per triangle: the packed kernel's loop over single points (966 of them)."""
    test_row_kinds(form, alpha, beta, 21, 24, 1)
