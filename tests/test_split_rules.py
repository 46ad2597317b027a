"""How the pair kernels cut their sources into slices (csrc/splits.h), compiled on its own with the host compiler (no
GPU): the rules' bounds over the point counts, at the GB300's 152 SMs."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
SRC = os.path.join(os.path.dirname(HERE), "paper_2108_10481_gb300", "csrc")
SMS = 152

DRIVER = r"""
#include <cstdio>
#include <cstdlib>
#include "splits.h"
using namespace pb;
int main(int argc, char** argv) {  // lo hi step
    for (long long np = atoll(argv[1]); np <= atoll(argv[2]); np += atoll(argv[3]))
        for (int mode = 0; mode < 2; ++mode)
            for (int kind = 0; kind < (mode ? 3 : 2); ++kind)
                for (int resident = 6; resident <= 9; resident += 3) {
                    const int slots = resident * %(sms)d;
                    const Pair64Plan p = pair64_plan(np, mode, kind, %(sms)d, slots);
                    const Pair64Plan o = pair64_one(np, mode, kind, %(sms)d, slots);
                    printf("%%lld %%d %%d %%d %%d %%.17g %%.17g\n", np, mode, kind, p.sym.nblock > 0, p.slices(), p.cost, o.cost);
                }
    return 0;
}
""" % {"sms": SMS}


def compile_driver(path, source):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no host C++ compiler")
    (path / "driver.cpp").write_text(source)
    subprocess.run([cxx, "-std=c++17", "-O1", "-I" + SRC, str(path / "driver.cpp"), "-o", str(path / "driver")], check=True)
    return str(path / "driver")


@pytest.fixture(scope="module")
def fp64_plans(tmp_path_factory):
    exe = compile_driver(tmp_path_factory.mktemp("fp64"), DRIVER)
    rows = []
    for rng in ((6, 4000, 6), (4002, 66000, 186), (62400, 64600, 6), (70000, 800000, 7302)):
        out = subprocess.run([exe, *map(str, rng)], check=True, capture_output=True, text=True).stdout
        rows += [[float(w) for w in line.split()] for line in out.splitlines()]
    return rows


def test_fp64_never_dearer_than_one_direction(fp64_plans):
    """At 62,465 to 64,512 points the both-directions kernel has one slice of rows: one direction is the cheaper."""
    for np_, mode, kind, both, slices, cost, one in fp64_plans:
        assert cost <= one, (np_, mode, kind)
        if np_ >= 62465:
            assert not both, (np_, mode, kind)
        if np_ <= 48000:
            assert both, (np_, mode, kind)


def test_fp64_slices_within_their_bounds(fp64_plans):
    for np_, mode, kind, both, slices, cost, one in fp64_plans:
        assert 1 <= slices <= 64
        assert slices <= 32 or slices * (10 if mode else 2) * np_ * 8 <= 32e6, (np_, mode, kind)


PACKED = r"""
#include <cstdio>
#include <cstdlib>
#include "splits.h"
using namespace pb;
int main(int argc, char** argv) {  // lo hi step: sources of a fast slice by launch shape, and by whole waves
    static const int shapes[4][2] = {{64, 1024}, {32, 1024}, {128, 1024}, {64, 512}};  // records per tile, targets per CTA
    for (long long np = atoll(argv[1]); np <= atoll(argv[2]); np += atoll(argv[3]))
        for (int mode = 0; mode < 2; ++mode)
            for (int k = 0; k < 4; ++k) {
                const int ts = shapes[k][0], tu = ts / 3 * 3;
                int S = x2_splits(np, shapes[k][1], ts, %(sms)d, x2_longest(np, mode, ts, %(sms)d));
                S = scaled_splits(S, 1.0, np, tu);
                const long long chunk = ((np + S - 1) / S + tu - 1) / tu * tu;
                const int W = choose_splits(np, 1024, ts, (mode ? 2 : 4) * %(sms)d);
                printf("%%lld %%d %%d %%d %%lld %%lld\n", np, mode, k, S, chunk, (long long)(((np + W - 1) / W + ts - 1) / ts * ts));
            }
    return 0;
}
""" % {"sms": SMS}


def test_fast_slices_no_longer_than_whole_waves(tmp_path):
    """The fast FP32 sums run over no more sources than the whole-wave rule's slices have, at any launch shape."""
    exe = compile_driver(tmp_path, PACKED)
    for rng in ((1, 4000, 1), (4002, 120000, 42)):
        out = subprocess.run([exe, *map(str, rng)], check=True, capture_output=True, text=True).stdout
        for line in out.splitlines():
            np_, mode, shape, S, chunk, wave = map(int, line.split())
            assert S <= 36
            assert chunk <= wave + (64, 32, 128, 64)[shape] // 2, line  # to the nearest tile


CAPPED = r"""
#include <cstdio>
#include <cstdlib>
#include "splits.h"
using namespace pb;
int main(int argc, char** argv) {  // lo hi step: bytes of every application's partial sums against a request's
    for (long long np = atoll(argv[1]); np <= atoll(argv[2]); np += atoll(argv[3]))
        for (int mixed = 0; mixed < 2; ++mixed)
            for (int least = 0; least < 2; ++least) {
                const double cap = least ? least_part_bytes(np, %(sms)d) : part_bytes(np, %(sms)d, mixed);
                double most = 0.0;
                for (int mode = 0; mode < 2; ++mode) {
                    const double sum = (double)np * (mode ? 10 : 2);
                    if (mixed)
                        for (int acc = 0; acc < 2; ++acc)
                            for (double scale = 0.5; scale <= 2.0; scale *= 2.0) {
                                const int n = capped_slices(cap, np, mode ? 10 : 2, acc ? 8 : 4);
                                int S = x2_splits(np, acc ? 512 : 1024, 64, %(sms)d, acc ? 0 : x2_longest(np, mode, 64, %(sms)d), n);
                                S = scaled_splits(S, scale, np, 63, n);
                                if (S * sum * (acc ? 8 : 4) > most) most = S * sum * (acc ? 8 : 4);
                            }
                    else
                        for (int kind = 0; kind < (mode ? 3 : 2); ++kind)
                            for (int resident = 6; resident <= 9; resident += 3) {
                                const Pair64Plan p = pair64_plan(np, mode, kind, %(sms)d, resident * %(sms)d, cap);
                                if (p.slices() * sum * 8 > most) most = p.slices() * sum * 8;
                            }
                }
                printf("%%lld %%d %%d %%.17g %%.17g\n", np, mixed, least, most, cap);
            }
    return 0;
}
""" % {"sms": SMS}


def test_partial_sums_within_a_request_s_bytes(tmp_path):
    """Served applications' partial sums, tuned split scales included, stay within what the server's budget counts."""
    exe = compile_driver(tmp_path, CAPPED)
    for rng in ((1, 4000, 7), (4002, 66000, 186), (62400, 64600, 6), (70000, 800000, 7302)):
        out = subprocess.run([exe, *map(str, rng)], check=True, capture_output=True, text=True).stdout
        for line in out.splitlines():
            np_, mixed, least, most, cap = (float(w) for w in line.split())
            assert 0 < most <= cap, line
