"""Reaction potential of more charges than one grid holds: 65,535 in FP64 (a block each) and 65,535 x 32 in split-coordinate
FP32. The potential at a charge does not depend on the others, so repeated positions give the oracle's values of the first
few. Tolerances as the charge sums' test (1e-12, 1e-6)."""
import numpy as np
import pytest

import oracle
from oracle import oracle as O
from synth.charges import ball_charges
from synth.icosphere import uv_ellipsoid
from tests.gpu_common import PHYS, rel

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,n_q,tol", [("f64", 65535, 1e-12), ("f64", 65537, 1e-12), ("f64", 140001, 1e-12),
                                          ("split", 16385, 1e-6), ("split", 65535 * 32, 1e-6),
                                          ("split", 65535 * 32 + 1, 1e-6), ("split", 4300003, 1e-6)])
def test_many_charges(prec, n_q, tol):
    import torch

    import paper_2108_10481_gb300 as pb
    v, t = uv_ellipsoid(13, 11, (2.0, 1.6, 1.3), center=(0.3, -0.2, 0.1), twist=0.15)
    xq, q = ball_charges(701, 0.9, 11)
    xq = xq + np.array([0.3, -0.2, 0.1])
    plan = {"far_q": 6, "n_ss": 2}
    nv = v.shape[0]
    x = np.random.default_rng(4).standard_normal(2 * nv)
    ref = oracle.reaction_potential(v, t, x[:nv], x[nv:], xq, O.Plan(**plan))
    ctx = pb.pb_init(0)
    m = pb.pb_mesh_load(ctx, v, t, **plan)
    P = pb.Params(PHYS.eps_int, PHYS.eps_ext, PHYS.kappa)
    reps = -(-n_q // 701)
    dxq, dq = (torch.as_tensor(a, device="cuda").repeat(*r)[:n_q].contiguous() for a, r in ((xq, (reps, 1)), (q, (reps,))))
    phi = torch.empty_like(dq)
    dg, _ = pb.pb_energy(ctx, m, torch.as_tensor(x, device="cuda"), "juffer", dxq, dq, P, phi=phi,
                         prec=pb.PB_F64 if prec == "f64" else pb.PB_F32_ACCURATE)
    want = np.tile(ref, reps)[:n_q]
    assert rel(phi.cpu().numpy(), want) < tol
    assert abs(dg - 0.5 * float(dq.cpu().numpy() @ want)) < tol * np.linalg.norm(dq.cpu().numpy()) * np.linalg.norm(want)
