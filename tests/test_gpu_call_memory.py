"""Device memory that calls need for themselves only: pb_energy leaves none with the mesh, a context gives back what it
kept when it is freed, and a server whose requests are done holds no more than when it was made (its budget counts what its
requests hold). Bounds: 2 MB, the device's allocation granularity; each of the calls needs 8 MB or more for itself."""
import numpy as np
import pytest

from synth import icosphere
from synth.charges import ball_charges

pytestmark = pytest.mark.gpu
SLACK = 2 << 20


def free_bytes():
    import torch
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]


def energy(pb, ctx, m, nv, prec):
    import torch
    xq, q = ball_charges(200, 4.0, 3)
    dxq, dq = torch.as_tensor(xq, device="cuda"), torch.as_tensor(q, device="cuda")
    x = torch.ones(2 * nv, dtype=torch.float64, device="cuda")
    pb.pb_energy(ctx, m, x, "juffer", dxq, dq, pb.Params(4.0, 80.0, 0.125), prec=prec)


@pytest.mark.parametrize("prec", ["f64", "split"])
def test_energy_leaves_nothing_with_the_mesh(prec):
    import paper_2108_10481_gb300 as pb
    v, t = icosphere(5, 9.0)  # 122,880 points
    ctx = pb.pb_init(0)
    meshes = [pb.pb_mesh_load(ctx, v, t, far_q=6, n_ss=2) for _ in range(3)]
    prec = pb.PB_F64 if prec == "f64" else pb.PB_F32_ACCURATE
    energy(pb, ctx, meshes[0], len(v), prec)
    held, free = [m.info()["device_bytes"] for m in meshes], free_bytes()
    for m in meshes:
        energy(pb, ctx, m, len(v), prec)
    assert [m.info()["device_bytes"] for m in meshes] == held
    assert free_bytes() >= free - SLACK


def test_a_freed_context_holds_nothing():
    import paper_2108_10481_gb300 as pb
    v, t = icosphere(3, 4.0)
    for k in range(2):  # the first time round loads the kernels
        free = free_bytes()
        ctx = pb.pb_init(0)
        m = pb.pb_mesh_load(ctx, v, t, far_q=6, n_ss=4)
        nf = pb.pb_near_build(ctx, m, 0.125)
        nf.free()
        m.free()
        ctx.free()
    assert free_bytes() >= free - SLACK


@pytest.mark.parametrize("precision", ["PB_F64", "PB_MIXED"])
def test_an_idle_server_holds_nothing(precision):
    import paper_2108_10481_gb300 as pb
    v, t = icosphere(3, 4.0)  # its near build needs 18 MB for itself
    xq, q = ball_charges(20, 1.5, 3)
    opts = pb.solve_opts(tol=1e-6, max_it=300, precision=getattr(pb, precision), inner_tol=1e-4)
    form, prec = pb.CASES[10]

    def serve(srv):
        pb.pb_submit(srv, v, t, xq, q, pb.Params(4.0, 80.0, 0.125), form, prec, opts=opts)
        done = []
        while not done:
            pb.pb_server_step(srv)
            done = pb.pb_poll(srv)
        assert done[0]["status"] == 0

    for k in range(2):  # the first time round loads the kernels
        ctx = pb.pb_init(0)
        free = free_bytes()
        srv = pb.pb_server_create(ctx, 1 << 30, 2)
        serve(srv)
        assert k == 0 or free_bytes() >= free - 2 * SLACK  # its own tables
        srv.free()
        ctx.free()
