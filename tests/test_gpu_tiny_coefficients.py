"""Combined forms whose alpha or beta is below FP32's (or FP64's) normal range: the result is that of the coefficient zero.
Tolerances: rounding of one precision's two loops, FP32 2e-5, split 2e-6, treecode 1e-4 (as the row kinds' test), FP64 1e-12."""
import pytest

from synth.icosphere import uv_ellipsoid

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("form", ["cfie_ext", "cfie_int"])
@pytest.mark.parametrize("tiny", [(1e-42, 0.5), (0.7, -1e-42), (1e-42, 1e-42), (1e-310, 0.5), (1e-30, 1e-20)])
def test_as_with_the_coefficient_zero(form, tiny):
    import torch

    import paper_2108_10481_gb300 as pb
    v, t = uv_ellipsoid(21, 24, (2.0, 1.6, 1.3), center=(0.3, -0.2, 0.1), twist=0.1)
    ctx = pb.pb_init(0)
    m = pb.pb_mesh_load(ctx, v, t, far_q=3, n_ss=3)
    nf = pb.pb_near_build(ctx, m, 0.125)
    P = pb.Params(4.0, 80.0, 0.125)
    x = torch.randn(2 * v.shape[0], dtype=torch.float64, device="cuda", generator=torch.Generator("cuda").manual_seed(1))
    zero = [c if abs(c) > 1e-10 else 0.0 for c in tiny]

    def apply(prec, alpha, beta):
        return pb.pb_system_apply(ctx, m, nf, P, form, x, prec=prec, alpha=alpha, beta=beta)

    for prec, tree, tol in ((pb.PB_F64, False, 1e-12), (pb.PB_F32, False, 2e-5), (pb.PB_F32_ACCURATE, False, 2e-6),
                            (pb.PB_F32, True, 1e-4)):
        pb.pb_set_treecode(ctx, tree, 6, 0.7, 0)
        ref = apply(prec, *zero)
        assert float((apply(prec, *tiny) - ref).norm() / ref.norm()) < tol, (prec, tree)
