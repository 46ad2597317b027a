"""Formula counts of the pair kernels' profile: flops per point pair of the FP64 kernel that runs (V/K rows and V/K + D/T
rows, both directions at once and, above 64,512 points, one), operations of the packed and of the scalar FP32 kernel."""
import os

import pytest

from synth.icosphere import uv_ellipsoid

pytestmark = pytest.mark.gpu


def counted(n_lat, form, prec, kernel):
    import torch

    import paper_2108_10481_gb300 as pb
    v, t = uv_ellipsoid(20, n_lat, (2.0, 1.6, 0.0633 * n_lat), twist=0.05)
    ctx = pb.pb_init(0)
    m = pb.pb_mesh_load(ctx, v, t, far_q=6, n_ss=2)
    nf = pb.pb_near_build(ctx, m, 0.125)
    pb.pb_set_treecode(ctx, False, 6, 0.7, 0)
    pb.pb_profile(ctx, True)
    pb.pb_system_apply(ctx, m, nf, pb.Params(4.0, 80.0, 0.125), form,
                       torch.ones(2 * len(v), dtype=torch.float64, device="cuda"), prec=getattr(pb, prec))
    torch.cuda.synchronize()
    r = pb.pb_profile_read(ctx, getattr(pb, kernel))
    np_ = m.info()["n_points"]
    assert r["launches"] == 1 and r["pairs"] == np_ * np_
    return r["ops"] / r["pairs"]


@pytest.mark.parametrize("n_lat,form,flops", [(17, "direct_int", 28.5), (17, "juffer", 48.0), (271, "direct_int", 43.0),
                                              (271, "juffer", 67.0)])
def test_fp64(n_lat, form, flops):
    assert counted(n_lat, form, "PB_F64", "PB_KERNEL_PAIR64") == pytest.approx(flops)


@pytest.mark.parametrize("scalar,ops", [(False, 29.667), (True, 36.0)])
def test_fp32(monkeypatch, scalar, ops):
    if scalar:
        monkeypatch.setitem(os.environ, "PBBEM_PAIR_KERNEL", "1")
    assert counted(17, "juffer", "PB_F32", "PB_KERNEL_PAIR32") == pytest.approx(ops)
