"""The split-coordinate kernels' sums over tiles (csrc/wide.h), compiled on its own with the host compiler (no GPU):
FP32 values added into three FP32 words against the exact sum. Bound: half an ulp of FP64, and 2^-71 a term of the largest
partial sum (lo's additions), which is below the error of FP64 accumulation; without the third word (about 48 bits) the
same sums miss it."""
import math
import os
import shutil
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
SRC = os.path.join(os.path.dirname(HERE), "paper_2108_10481_gb300", "csrc")

DRIVER = r"""
#include <cstdio>
#include "wide.h"
struct Ops {
    static float add(float a, float b) { volatile float r = a + b; return r; }
    static float sub(float a, float b) { volatile float r = a - b; return r; }
};
int main() {
    float b, hi = 0, mid = 0, lo = 0, hi2 = 0, mid2 = 0;
    while (fread(&b, 4, 1, stdin) == 1) {
        pb::wide_add<Ops>(hi, mid, lo, b);
        float none = 0;
        pb::wide_add<Ops>(hi2, mid2, none, b);  // the third word thrown away
    }
    printf("%.17g %.17g\n", pb::wide_value(hi, mid, lo), pb::wide_value(hi2, mid2, 0.0f));
    return 0;
}
"""


@pytest.fixture(scope="module")
def sums(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no host C++ compiler")
    d = tmp_path_factory.mktemp("wide")
    (d / "driver.cpp").write_text(DRIVER)
    subprocess.run([cxx, "-std=c++17", "-O1", "-I" + SRC, str(d / "driver.cpp"), "-o", str(d / "driver")], check=True)

    def run(values):
        out = subprocess.run([str(d / "driver")], input=np.asarray(values, np.float32).tobytes(), check=True,
                             capture_output=True).stdout.split()
        return [float(w) for w in out]

    return run


def bound(values):
    exact = math.fsum(float(b) for b in values)
    peak = float(np.abs(np.cumsum(np.asarray(values, np.float64))).max())
    return exact, 2.0 ** -53 * abs(exact) + len(values) * 2.0 ** -71 * peak


@pytest.mark.parametrize("n", [1, 2, 46, 976, 10500])
@pytest.mark.parametrize("kind", ["positive", "signed", "spread", "cancelling", "tiny"])
def test_no_fewer_bits_than_fp64(sums, n, kind):
    rng = np.random.default_rng(n)
    b = np.float32(rng.uniform(0.1, 1.0, n) if kind == "positive" else rng.standard_normal(n))
    if kind == "spread":
        b = np.float32(b * 10.0 ** rng.uniform(-8.0, 0.0, n))
    if kind == "cancelling":  # a sum a thousandth of its largest partial sums
        b = np.concatenate([np.float32(1e3) + b, np.float32(-1e3) + b[::-1]])
    if kind == "tiny":
        b = np.float32(b * 1e-36)
    exact, tol = bound(b)
    assert abs(sums(b)[0] - exact) <= tol


def test_two_words_miss_the_bound(sums):
    rng = np.random.default_rng(3)
    b = np.float32(rng.uniform(0.1, 1.0, 10500) * 10.0 ** rng.uniform(-8.0, 0.0, 10500))
    exact, tol = bound(b)
    assert abs(sums(b)[1] - exact) > 4 * tol


def test_past_the_range(sums):
    assert sums([3e38, 3e38])[0] == math.inf
    assert math.isnan(sums([math.inf, -math.inf])[0])
    assert math.isnan(sums([1.0, math.nan])[0])
