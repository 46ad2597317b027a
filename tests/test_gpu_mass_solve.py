"""Mass preconditioner against a dense solve with the closed-form P1 mass matrix: the smallest closed surface, vertex
counts around the 2,048 up to which one cluster runs the whole iteration, rows longer than those held in registers
(poles), and the scaled form. FP64: 34 Chebyshev steps, rounding level (1e-13); FP32 count: 16 steps, 2/3^16 = 4.6e-8 in
the norm of the matrix's diagonal, the one compared in (5e-8)."""
import numpy as np
import pytest

from synth.icosphere import uv_ellipsoid

pytestmark = pytest.mark.gpu


# 5, 50, 2,046, 2,048, 2,049 and 2,050 vertices; poles of 3 to 62 triangles
@pytest.mark.parametrize("n_lon,n_lat", [(3, 2), (12, 5), (28, 74), (62, 34), (23, 90), (32, 65)])
@pytest.mark.parametrize("precond", ["mass", "scaled_mass"])
def test_mass_solve(n_lon, n_lat, precond):
    import torch

    import paper_2108_10481_gb300 as pb
    v, t = uv_ellipsoid(n_lon, n_lat, (2.0, 1.6, 1.8 * n_lat / n_lon), twist=0.05)
    nv = v.shape[0]
    p = v[t]
    area = 0.5 * np.linalg.norm(np.cross(p[:, 1] - p[:, 0], p[:, 2] - p[:, 0]), axis=1)
    M = np.zeros((nv, nv))
    for a in range(3):
        for b in range(3):
            np.add.at(M, (t[:, a], t[:, b]), area / (6.0 if a == b else 12.0))
    x = np.random.default_rng(1).standard_normal(2 * nv)
    sa, sb = (1.0 + 80.0 / 4.0, 1.0 + 4.0 / 80.0) if precond == "scaled_mass" else (1.0, 1.0)
    ref = np.concatenate([np.linalg.solve(M, x[:nv]) / sa, np.linalg.solve(M, x[nv:]) / sb])
    ctx = pb.pb_init(0)
    m = pb.pb_mesh_load(ctx, v, t, far_q=1, n_ss=2)
    nf = pb.pb_near_build(ctx, m, 0.125)
    w = np.sqrt(np.tile(np.diag(M), 2))
    for prec, tol in ((pb.PB_F64, 1e-13), (pb.PB_F32, 5e-8)):
        y = pb.pb_precond_apply(ctx, m, nf, pb.Params(4.0, 80.0, 0.125), "juffer", precond,
                                torch.as_tensor(x, device="cuda"), prec=prec).cpu().numpy()
        for half in (slice(0, nv), slice(nv, None)):
            assert np.linalg.norm((w * (y - ref))[half]) < tol * np.linalg.norm((w * ref)[half])
