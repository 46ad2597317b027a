"""Split-coordinate pair sums where a CTA adds a hundred tiles and more (61,440 points): V/K rows and each kind of V/K +
D/T rows against the library's FP64 application. Tolerance 2e-7: a tile's 63 FP32 sums round at 2^-24 each and their errors
average out over the tiles; a lost or misplaced word of the sums over the tiles is orders above. The fast variant's launch
shape above 16,384 points (the row kinds' test has the one below), tolerance as there."""
import pytest

from synth import icosphere
from tests.test_gpu_pair32_kinds import FORMS

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def case():
    import torch

    import paper_2108_10481_gb300 as pb
    v, t = icosphere(5, 9.0)
    ctx = pb.pb_init(0)
    m = pb.pb_mesh_load(ctx, v, t, far_q=3, n_ss=3)
    assert m.info()["n_points"] == 61440
    nf = pb.pb_near_build(ctx, m, 0.125)
    x = torch.as_tensor(1.0 + 0.3 * v[:, 2] / 9.0, device="cuda").repeat(2)
    return pb, ctx, m, nf, x


@pytest.mark.parametrize("form,alpha,beta", FORMS)
def test_many_tiles(case, form, alpha, beta):
    pb, ctx, m, nf, x = case
    P = pb.Params(4.0, 80.0, 0.125)

    def apply(prec):
        return pb.pb_system_apply(ctx, m, nf, P, form, x, prec=prec, alpha=alpha, beta=beta)

    ref = apply(pb.PB_F64)
    assert float((apply(pb.PB_F32_ACCURATE) - ref).norm() / ref.norm()) < 2e-7


@pytest.mark.parametrize("form,alpha,beta", FORMS)
def test_fast_variant(case, form, alpha, beta):
    pb, ctx, m, nf, x = case
    P = pb.Params(4.0, 80.0, 0.125)
    pb.pb_set_treecode(ctx, False, 6, 0.7, 0)

    def apply(prec):
        return pb.pb_system_apply(ctx, m, nf, P, form, x, prec=prec, alpha=alpha, beta=beta)

    ref = apply(pb.PB_F64)
    assert float((apply(pb.PB_F32) - ref).norm() / ref.norm()) < 2e-5
