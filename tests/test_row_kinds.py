"""The rule that picks a loop of the pair kernels and the treecode for a block operator's coefficients (csrc/kinds.h),
compiled on its own with the host compiler (no GPU). Coefficients in the order of a kernel row: Laplace and Yukawa of
V, K and of D, T (or V, K again)."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
SRC = os.path.join(os.path.dirname(HERE), "paper_2108_10481_gb300", "csrc")

DRIVER = r"""
#include <cstdio>
#include <cstdlib>
#include "kinds.h"
int main(int, char** argv) {
    const int mode = atoi(argv[1]);
    double k[2][4];
    for (int q = 0; q < 8; ++q) k[q / 4][q % 4] = atof(argv[2 + q]);
    int lrow = -1;
    const int t = pb::tree_kind(mode, k, &lrow);
    printf("%d %d %d %d\n", pb::pair64_kind(mode, k), pb::pair32_kind(mode, k), t, lrow);
    return 0;
}
"""

TINY = 1e-42  # below FP32's normal range
# mode, coefficients, kinds of the FP64 and FP32 pair kernels and the treecode, row without a Yukawa term (V/K rows)
CASES = [
    (0, (1, 0, -1, 0, 0, .05, 0, 1), (0, 0, 3, 0)),             # direct form
    (0, (0, .05, 0, 1, 1, 0, -1, 0), (0, 0, 3, 1)),             # its rows exchanged
    (0, (1, 0, -1, 0, 0, 0, 0, 0), (1, 0, 3, 0)),               # Laplace only
    (0, (1, 1, -1, 1, 1, 0, -1, 0), (0, 0, 0, 1)),              # both in a row
    (1, (1, -1, -1, 1, 1, -.05, 1, -1), (2, 2, 2, None)),       # both kernels everywhere
    (1, (1, 0, -1, 0, 1, 0, 1, 0), (1, 1, 1, None)),            # no Yukawa term
    (1, (1, 0, 0, 0, 1, 0, 1, 0), (1, 1, 0, None)),             # ... nor a K: the dipoles carry no coefficient
    (1, (0, 1, 0, 1, 1, -.05, 1, -1), (0, 0, 0, None)),         # a row without Laplace terms
    (1, (TINY, -1, -TINY, 1, 1, -.05, 1, -1), (0, 0, 0, None)), # ... or as good as without
    (1, (1, -1, -1, 1, 1, -.05, 1e-310, -1), (0, 0, 0, None)),
    (1, (1, -1, -1e15, 1, 1, -.05, 1, -1), (0, 0, 0, None)),
    (1, (1, -1e15, -1, 1, 1, -.05, 1, -1), (0, 0, 0, None)),
    (1, (1, 0, -TINY, 0, 1, 0, 1, 0), (1, 1, 0, None)),
    (1, (1, TINY, -1, TINY, 1, TINY, 1, TINY), (2, 2, 2, None)),  # small Yukawa terms are no trouble
    (1, (1, -1, float("nan"), 1, 1, -.05, 1, -1), (0, 0, 0, None)),
]


@pytest.fixture(scope="module")
def driver(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no host C++ compiler")
    d = tmp_path_factory.mktemp("kinds")
    (d / "driver.cpp").write_text(DRIVER)
    subprocess.run([cxx, "-std=c++17", "-O1", "-I" + SRC, str(d / "driver.cpp"), "-o", str(d / "driver")], check=True)
    return str(d / "driver")


@pytest.mark.parametrize("mode,k,want", CASES)
def test_kind(driver, mode, k, want):
    out = subprocess.run([driver, str(mode), *map(repr, map(float, k))], check=True, capture_output=True, text=True).stdout
    got = tuple(map(int, out.split()))
    assert got[:3] == want[:3]
    assert mode == 1 or got[3] == want[3]
