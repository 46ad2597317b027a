"""Right-hand side and reaction potential against the oracle's charge sums: one charge, counts around the blocks of 32
and tiles of 256, each far rule (blocks of whole triangles), a band plan, both precisions. Tolerances: FP64 1e-12;
split-coordinate FP32 1e-6 (about 1e-7 by the declaration)."""
import numpy as np
import pytest

import oracle
from oracle import oracle as O
from synth.charges import ball_charges
from synth.icosphere import uv_ellipsoid
from tests.gpu_common import PHYS, rel

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_q", [1, 31, 33, 257, 700])
@pytest.mark.parametrize("plan", [{"far_q": 6, "n_ss": 2}, {"far_q": 3, "n_ss": 2}, {"far_q": 1, "n_ss": 2},
                                  {"far_q": 3, "n_ss": 2, "band_eta": 2.0, "band_q": 6}])
def test_charge_sums(n_q, plan):
    import torch

    import paper_2108_10481_gb300 as pb
    v, t = uv_ellipsoid(13, 11, (2.0, 1.6, 1.3), center=(0.3, -0.2, 0.1), twist=0.15)  # 260 triangles
    xq, q = ball_charges(n_q, 0.9, 11)
    xq = xq + np.array([0.3, -0.2, 0.1])
    pl = O.Plan(**plan)
    bD, bN = oracle.source_projections(v, t, xq, q, PHYS.eps_int, pl)
    nv = v.shape[0]
    x = np.random.default_rng(4).standard_normal(2 * nv)
    ref = oracle.reaction_potential(v, t, x[:nv], x[nv:], xq, pl)
    ctx = pb.pb_init(0)
    m = pb.pb_mesh_load(ctx, v, t, **plan)
    P = pb.Params(PHYS.eps_int, PHYS.eps_ext, PHYS.kappa)
    dxq, dq, dx = (torch.as_tensor(a, device="cuda") for a in (xq, q, x))
    for prec, tol in ((pb.PB_F64, 1e-12), (pb.PB_F32_ACCURATE, 1e-6)):
        rhs = pb.pb_rhs_charges(ctx, m, dxq, dq, P, "juffer", prec=prec).cpu().numpy()
        assert rel(rhs, np.concatenate([bD, bN])) < tol
        phi = torch.empty_like(dq)
        for _ in range(2):  # the second call finds its workspace
            dg, _ = pb.pb_energy(ctx, m, dx, "juffer", dxq, dq, P, phi=phi, prec=prec)
            assert rel(phi.cpu().numpy(), ref) < tol
            assert abs(dg - 0.5 * q @ ref) < tol * np.linalg.norm(q) * np.linalg.norm(ref)
