"""FP64 double-layer operators against the oracle's sums in the compiler's long double (64 or more bits of mantissa): the
near field's subtraction of the far rule has to cancel what the pair kernel adds, down to rounding. Tolerance three unit
roundoffs (3.3e-16) of the result's norm: independent roundings of the terms leave one to two; an error common to a
triangle's points does not average out."""
import ctypes
import os
import re
import subprocess

import numpy as np
import pytest

from oracle import oracle as O
from synth.icosphere import uv_ellipsoid
from tests.gpu_common import OPS

pytestmark = pytest.mark.gpu
SRC = os.path.join(os.path.dirname(os.path.abspath(O.__file__)), "bem_oracle.c")
LD = np.longdouble


@pytest.fixture(scope="module")
def wide_oracle(tmp_path_factory):
    text = open(SRC).read()
    for a, b in ((r"\bdouble\b", "long double"), (r"\bsqrt\(", "sqrtl("), (r"\bexp\(", "expl("),
                 (r"3\.14159265358979323846", "3.14159265358979323846264338327950288L")):
        text = re.sub(a, b, text)
    d = tmp_path_factory.mktemp("oracle")
    (d / "wide.c").write_text(text)
    subprocess.run(["gcc", "-O2", "-ffp-contract=off", "-fPIC", "-shared", "-fopenmp", "-std=c11", str(d / "wide.c"), "-o",
                    str(d / "wide.so"), "-lm"], check=True)
    lib = ctypes.CDLL(str(d / "wide.so"))
    P, I64, I, D = ctypes.c_void_p, ctypes.c_int64, ctypes.c_int, ctypes.c_longdouble
    lib.oracle_assemble_dense.argtypes = [P, I64, P, I64, I, P, P, P, P, P, D, D, I, P, P, I] + [P] * 7

    def double_layers(v, t, kappa, plan):
        rl, rw, ng, gx, gw = O._rules(plan)
        eta, nb, bl, bw = O._band(plan)
        v, rl, rw, gx, gw, bl, bw = (np.ascontiguousarray(a, dtype=LD) for a in (v, rl, rw, gx, gw, bl, bw))
        t = np.ascontiguousarray(t, dtype=np.int32)
        mats = [np.zeros((len(v), len(v)), dtype=LD) for _ in range(7)]
        lib.oracle_assemble_dense(v.ctypes.data, len(v), t.ctypes.data, len(t), len(rl), rl.ctypes.data, rw.ctypes.data,
                                  ng.ctypes.data, gx.ctypes.data, gw.ctypes.data, kappa, eta, nb, bl.ctypes.data,
                                  bw.ctypes.data, 0, *[m.ctypes.data for m in mats])
        return {"KL": mats[1], "TL": mats[1].T, "KY": mats[4], "TY": mats[4].T}

    return double_layers


@pytest.mark.parametrize("plan", [{"far_q": 6, "n_ss": 4}, {"far_q": 3, "n_ss": 4},
                                  {"far_q": 3, "n_ss": 4, "band_eta": 3.0, "band_q": 6, "n_ss_coin": 3}])
def test_double_layers_to_rounding(wide_oracle, plan):
    import torch

    import paper_2108_10481_gb300 as pb
    v, t = uv_ellipsoid(13, 12, (2.0, 1.7, 1.5), center=(0.3, -0.2, 0.1), twist=0.15)
    ops = wide_oracle(v, t, 0.125, O.Plan(**plan))
    ctx = pb.pb_init(0)
    m = pb.pb_mesh_load(ctx, v, t, **plan)
    nf = pb.pb_near_build(ctx, m, 0.125)
    x = 1.0 + 0.3 * v[:, 2] + 0.2 * v[:, 0] * v[:, 1]
    for name, mat in ops.items():
        op, kern = OPS[name]
        y = pb.pb_op_apply(ctx, m, nf, op, kern, pb.PB_F64, torch.as_tensor(x, device="cuda")).cpu().numpy()
        ref = mat @ x.astype(LD)
        err = float(np.sqrt(((y.astype(LD) - ref) ** 2).sum() / (ref ** 2).sum()))
        print(name, plan, "%.2e" % err)
        assert err < 3.3e-16, (name, err)
