"""Near field of adjacent and band pairs against the oracle over what selects its code path: the lanes per pair (few or many
pairs), the degree of the Yukawa polynomials (kappa times the triangles' size, past their range the exponentials), the
singular order, the far rule and the band's rules. One FP64 application per operator; tolerance as the operator parity tests (1e-12)."""
import numpy as np
import pytest

import oracle
from .gpu_common import OPS, rel
from oracle import oracle as O
from synth import icosphere
from synth.icosphere import uv_ellipsoid

pytestmark = pytest.mark.gpu


def check(v, t, kappa, plan):
    import torch

    import paper_2108_10481_gb300 as pb
    ref = oracle.assemble(v, t, kappa, O.Plan(**plan))
    ctx = pb.pb_init(0)
    m = pb.pb_mesh_load(ctx, v, t, **plan)
    nf = pb.pb_near_build(ctx, m, kappa)
    x = np.random.default_rng(5).standard_normal(v.shape[0])
    dx = torch.as_tensor(x, device="cuda")
    for name in ("VL", "KL", "DL", "VY", "KY", "TY", "DY"):
        op, kern = OPS[name]
        y = pb.pb_op_apply(ctx, m, nf, op, kern, pb.PB_F64, dx).cpu().numpy()
        assert rel(y, getattr(ref, name) @ x) < 1e-12, (name, kappa, plan)
    nf.free()
    m.free()


@pytest.mark.parametrize("kappa", [0.0, 0.01, 0.125, 0.3, 0.45, 2.0])
def test_yukawa_sums_at_every_degree(kappa):
    v, t = icosphere(2, 2.0)
    check(v, t, kappa, {"far_q": 6, "n_ss": 4})


@pytest.mark.parametrize("plan", [{"far_q": 3, "n_ss": 3}, {"far_q": 1, "n_ss": 2}, {"far_q": 6, "n_ss": 5},
                                  {"far_q": 3, "n_ss": 4, "n_ss_coin": 1, "n_ss_edge": 3, "n_ss_vert": 6}])
def test_orders_and_far_rules(plan):
    v, t = uv_ellipsoid(9, 8, (2.0, 1.6, 1.3), center=(0.3, -0.2, 0.1), twist=0.15)
    check(v, t, 0.125, plan)


@pytest.mark.parametrize("far_q,band_q,eta", [(3, 6, 2.0), (1, 6, 1.5), (1, 3, 6.0)])
@pytest.mark.parametrize("n_lon,n_lat", [(9, 8), (31, 29)])
def test_band_rules(n_lon, n_lat, far_q, band_q, eta):
    v, t = uv_ellipsoid(n_lon, n_lat, (2.0, 1.6, 1.3), center=(0.3, -0.2, 0.1), twist=0.15)
    check(v, t, 0.125, {"far_q": far_q, "n_ss": 3, "band_eta": eta, "band_q": band_q})


@pytest.mark.parametrize("n_lon,n_lat,length", [(31, 29, 2.3), (20, 190, 14.0)])
def test_many_pairs(n_lon, n_lat, length):
    """1,736 triangles (4 lanes per vertex pair, a warp per edge pair) and 7,560 (4 and 8 lanes)."""
    v, t = uv_ellipsoid(n_lon, n_lat, (1.5, 1.4, length), twist=0.05)
    check(v, t, 0.125, {"far_q": 3, "n_ss": 4})


def test_rows_too_long_for_a_full_batch():
    """3,762 vertices, every pair of triangles in the band: rows of 3,762 entries, which leave room for 32 staged
    contributions a warp only. Rows of M, V_L and D_Y against the oracle's."""
    import torch

    import paper_2108_10481_gb300 as pb
    v, t = uv_ellipsoid(80, 48, (2.0, 1.6, 1.3), twist=0.02)
    plan = {"far_q": 1, "n_ss": 2, "band_eta": 64.0, "band_q": 3}
    rows = np.array([0, 5, 1900, v.shape[0] - 1])
    ref = oracle.assemble_rows(v, t, rows, 0.125, O.Plan(**plan))
    ctx = pb.pb_init(0)
    m = pb.pb_mesh_load(ctx, v, t, **plan)
    nf = pb.pb_near_build(ctx, m, 0.125)
    x = np.random.default_rng(6).standard_normal(v.shape[0])
    for name in ("M", "VL", "DY"):
        op, kern = OPS[name]
        y = pb.pb_op_apply(ctx, m, nf, op, kern, pb.PB_F64, torch.as_tensor(x, device="cuda")).cpu().numpy()
        assert rel(y[rows], ref[name] @ x) < 1e-12, name
