"""FP64 applications where the both-directions kernel gives way to the one-direction one: 62,400 points (61 blocks of
1,024), 63,360 (62, one block of rows an SM) and 64,560 (64). V/K and D/T rows against the oracle's at a few vertices;
tolerance as the FP64 operator parity tests (1e-12)."""
import numpy as np
import pytest

import oracle
from oracle import oracle as O
from synth.icosphere import uv_ellipsoid
from tests.gpu_common import OPS, PHYS, rel

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_lat,points", [(261, 62400), (265, 63360), (270, 64560)])
def test_rows_around_the_switch(n_lat, points):
    import torch

    import paper_2108_10481_gb300 as pb
    v, t = uv_ellipsoid(20, n_lat, (2.0, 1.6, 0.0633 * n_lat), twist=0.05)
    ctx = pb.pb_init(0)
    m = pb.pb_mesh_load(ctx, v, t, far_q=6, n_ss=3)
    assert m.info()["n_points"] == points
    nf = pb.pb_near_build(ctx, m, PHYS.kappa)
    rows = np.array([0, 7, 1500, 5000, v.shape[0] - 1])
    ops = oracle.assemble_rows(v, t, rows, PHYS.kappa, O.Plan(6, 3))
    x = np.random.default_rng(3).standard_normal(v.shape[0])
    for name in ("VL", "KL", "KY", "DY"):
        op, kern = OPS[name]
        y = pb.pb_op_apply(ctx, m, nf, op, kern, pb.PB_F64, torch.as_tensor(x, device="cuda")).cpu().numpy()
        assert rel(y[rows], ops[name] @ x) < 1e-12, name
