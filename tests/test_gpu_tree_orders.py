"""Treecode applications at every interpolation order, V/K rows and V/K + D/T rows, against the FP64 application.

Tolerance: a box seen under theta has its half width h at most theta times the distance, so the kernel as a function of
one coordinate is analytic within a Bernstein ellipse of t = 1 / theta = 2, rho = t + sqrt(t^2 - 1) = 3.73, and its
Chebyshev interpolant of degree p is within 4 / (rho - 1) rho^-p of it (relative to its size on the ellipse), three times
that for three axes: 4.4 rho^-p. Two more orders should give a factor rho^2 = 14; at least 1 / 0.6 is required, or the
2e-5 of an FP32 application reached."""
import pytest

from synth.icosphere import icosphere

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("form", ["juffer", "pmchwt_ext"])
@pytest.mark.parametrize("level,far_q", [(3, 3), (4, 6)])  # 3,840 and 30,720 points: direct sums alone, and several heights of slots
def test_orders(form, level, far_q):
    import torch

    import paper_2108_10481_gb300 as pb
    v, t = icosphere(level, 4.0)
    ctx = pb.pb_init(0)
    m = pb.pb_mesh_load(ctx, v, t, far_q=far_q, n_ss=3)
    nf = pb.pb_near_build(ctx, m, 0.125)
    P = pb.Params(4.0, 80.0, 0.125)
    w = torch.as_tensor(v, device="cuda", dtype=torch.float64) / 4.0
    x = torch.cat([1.0 + w[:, 0] + 0.5 * w[:, 1] * w[:, 2], 1.0 - w[:, 2] + w[:, 0] ** 2])
    ref = pb.pb_system_apply(ctx, m, nf, P, form, x, prec=pb.PB_F64)
    err = {}
    for order in range(2, 8):
        pb.pb_set_treecode(ctx, True, order, 0.5, 0)
        y = pb.pb_system_apply(ctx, m, nf, P, form, x, prec=pb.PB_F32)
        err[order] = float((y - ref).norm() / ref.norm())
    print(form, level, err)
    assert level == 3 or pb.pb_tree_info(m)["proxy_pairs"] > 0  # at level 3 no two clusters are far enough apart
    for order, e in err.items():
        assert e < max(4.4 * 3.73 ** -order, 2e-5), (order, err)
        if order > 3:
            assert e < max(0.6 * err[order - 2], 2e-5), (order, err)
