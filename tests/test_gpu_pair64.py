"""FP64 pair kernels (both directions of a pair at once up to 65,536 points, else one): every kind of row pair they have their own loop for (V/K rows with and without a Yukawa term; V/K + D/T
rows with any coefficients, without a Yukawa term, with both kernels everywhere), at point counts around the
kernels' blocks and chunks and at strong screening, against the oracle's dense operators. Tolerance as the FP64 operator
parity tests (1e-12 of the result, for the system forms of its largest block's result)."""
import numpy as np
import pytest

import oracle
from oracle import oracle as O
from synth import icosphere
from synth.icosphere import uv_ellipsoid
from tests.gpu_common import OPS, PHYS, rel

pytestmark = pytest.mark.gpu


def load(v, t, kappa, **plan):
    import paper_2108_10481_gb300 as pb
    ctx = pb.pb_init(0)
    m = pb.pb_mesh_load(ctx, v, t, **plan)
    return pb, ctx, m, pb.pb_near_build(ctx, m, kappa)


# 6, 64, 128, 132, 126, 420, 1,980, 8,976, 17,460 and 45,360 points (the last two: blocks of 512 and 1,024)
@pytest.mark.parametrize("n_lon,n_lat,far_q", [(3, 2, 1), (4, 9, 1), (8, 9, 1), (11, 7, 1), (7, 4, 3), (5, 8, 6),
                                               (11, 31, 3), (22, 35, 6), (30, 98, 3), (20, 190, 6)])
@pytest.mark.parametrize("form", ["direct_int", "juffer", "cfie_ext"])
def test_forms_at_ragged_sizes(n_lon, n_lat, far_q, form):
    import torch
    v, t = uv_ellipsoid(n_lon, n_lat, (2.0, 1.6, 1.3 * n_lat / n_lon), twist=0.1)
    pb, ctx, m, nf = load(v, t, PHYS.kappa, far_q=far_q, n_ss=3)
    ops = oracle.assemble(v, t, PHYS.kappa, O.Plan(far_q, 3))
    z = np.zeros(v.shape[0])
    # cfie_ext with alpha = 0: the first row without Laplace terms
    a, b = (0.0, 0.5) if form == "cfie_ext" else (0.0, 0.0)
    A, _ = O.system(form, ops, PHYS, z, z, *((a, b) if form == "cfie_ext" else ()))
    x = np.random.default_rng(2).standard_normal(A.shape[0])
    y = pb.pb_system_apply(ctx, m, nf, pb.Params(PHYS.eps_int, PHYS.eps_ext, PHYS.kappa), form,
                           torch.as_tensor(x, device="cuda"), alpha=a, beta=b).cpu().numpy()
    assert rel(y, A @ x) < 1e-12


@pytest.mark.parametrize("kappa", [0.0, 0.125, 40.0, 400.0])
def test_single_operators_and_screening(kappa):
    import torch
    v, t = icosphere(1, 2.0)
    pb, ctx, m, nf = load(v, t, kappa, far_q=6, n_ss=4)
    ops = oracle.assemble(v, t, kappa, O.Plan(6, 4))
    x = np.random.default_rng(3).standard_normal(v.shape[0])
    for name in ("VL", "KL", "TL", "DL", "VY", "KY", "TY", "DY"):
        op, kern = OPS[name]
        y = pb.pb_op_apply(ctx, m, nf, op, kern, pb.PB_F64, torch.as_tensor(x, device="cuda")).cpu().numpy()
        assert rel(y, getattr(ops, name) @ x) < 1e-12, name


def test_one_direction_at_a_time_beyond_the_symmetric_kernel():
    """75,600 points (more than 64 blocks of 1,024): V and T rows against the oracle's at a few vertices."""
    import torch
    v, t = uv_ellipsoid(20, 316, (2.0, 1.6, 20.0), twist=0.05)
    pb, ctx, m, nf = load(v, t, PHYS.kappa, far_q=6, n_ss=3)
    assert m.info()["n_points"] > 65536
    rows = np.array([0, 7, 1500, 6000, v.shape[0] - 1])
    ops = oracle.assemble_rows(v, t, rows, PHYS.kappa, O.Plan(6, 3))
    x = np.random.default_rng(3).standard_normal(v.shape[0])
    for name in ("VL", "KY", "DY"):
        op, kern = OPS[name]
        y = pb.pb_op_apply(ctx, m, nf, op, kern, pb.PB_F64, torch.as_tensor(x, device="cuda")).cpu().numpy()
        assert rel(y[rows], ops[name] @ x) < 1e-12, name
