"""The fixed-point softplus, sigmoid and sp'' of the FP64 element kernel (csrc/gd_fixed.cuh, which
compiles for the host) against long double, over the range of FP64 arguments.  Each keeps its
relative accuracy: the table path is off by a few 2^-58 where softplus and sigmoid are above 2^-5.1 (1 -
sigmoid, of positive arguments, is held to that absolute error like FP64's 1 - sigmoid is to 2^-53), the
tail's series by 2^-56, exp by 2^-56, and the conversion rounds to 2^-53; the bar is 4 2^-53.  As an operand of a layer product (units of 2^-56, 2^-62 for the sigmoid, of the scale
of the point's largest) each is off by half a unit (sigmoid: one) and that rounding."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2604_03411_gb300", "csrc")
CUDA = "/usr/local/cuda/include"

SOURCE = r"""
#include "gd_fixed.cuh"
#include <cstdio>
#include <cmath>
#include <random>
using namespace gd::fx;
typedef long double ld;
template <bool TAIL>
void check(double least)
{
    const double cut[] = {-745, -300, -129, -127.5, -64, -37, -10, -6.2, -3.4657359, -2.5, -1, -0.125, 0, 0.125, 1, 6.3, 37, 63.99};
    const ld bar = 4 * ldexpl(1.0L, -53);
    std::mt19937_64 g(1);
    for (int c = 0; c + 1 < (int)(sizeof cut / sizeof *cut); ++c) {
        if (cut[c] < least) continue;
        std::uniform_real_distribution<double> U(cut[c], cut[c + 1]);
        ld worst[5] = {0, 0, 0, 0, 0};
        for (int k = 0; k < 100000; ++k) {
            const double h = k ? U(g) : cut[c];
            const Act r = activation<TAIL>(h);
            const ld E = expl(-fabsl((ld)h)), sp = (h > 0 ? (ld)h : 0) + log1pl(E), sg = h < 0 ? E / (1 + E) : 1 / (1 + E);
            const ld dd = E / (1 + E) / (1 + E);
            if (sp < 1e-290L) continue;
            const double s = softplus_value(h, r), a = to_double(r.g, -62 - r.n), d = to_double(mulhi_s(r.g, r.c), -60 - r.n);
            const int hi = (int)(bits_of(h) >> 32);
            const int ep = TAIL ? softplus_exp_tail(order_key(hi)) : softplus_exp(hi > 0 ? hi : 0), es = ep < 0 ? ep : 0;
            const ld x = ldexpl((ld)softplus_operand(h, r, ep), ep - 56), y = ldexpl((ld)sigmoid_factor<TAIL>(r, es), es - 62);
            if (ep > -1000 && sp > ldexpl(1.0L, ep) * (1 + 1e-5L)) worst[3] = 9;       // the scale bounds the operand
            const bool scaled = ep > -1000;                               // below, every operand is 0
            const ld e[5] = {fabsl(s / sp - 1) / bar, fabsl(a / sg - 1) / bar, h > 2 ? fabsl(d - dd) / ldexpl(1.0L, -53) : fabsl(d / dd - 1) / bar,
                             scaled ? fabsl(x - sp) / (ldexpl(1.0L, ep - 57) + bar * sp) : 0,
                             scaled ? fabsl(y - sg) / (ldexpl(1.0L, es - 62) + bar * sg) : 0};
            for (int i = 0; i < 5; ++i) worst[i] = fmaxl(worst[i], e[i]);
        }
        printf("%g", cut[c]);
        for (ld w : worst) printf(" %.3f", (double)w);
        printf("\n");
    }
    if (!TAIL) return;
    const double far[] = {-1e3, -1e300, -INFINITY};
    for (double h : far) {
        const Act r = activation<TAIL>(h);
        if (softplus_value(h, r) != 0 || to_double(r.g, -62 - r.n) != 0 || to_double(mulhi_s(r.g, r.c), -60 - r.n) != 0) printf("%g 9\n", h);
    }
    if (softplus_value(70.5, activation<TAIL>(70.5)) != 70.5) printf("70.5 9\n");
}
int main()
{
    check<true>(-745);
    check<false>(-3.4657359);
    return 0;
}
"""


def test_activations_against_long_double(tmp_path):
    if not shutil.which("g++") or not os.path.exists(os.path.join(CUDA, "cuda_runtime.h")):
        pytest.skip("needs g++ and the CUDA headers")
    src, exe = tmp_path / "act.cpp", tmp_path / "act"
    src.write_text(SOURCE)
    subprocess.run(["g++", "-std=c++17", "-O2", "-x", "c++", "-I", CUDA, "-I", CSRC, str(src), "-o", str(exe)], check=True)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout
    rows = [[float(v) for v in line.split()] for line in out.splitlines()]
    assert len(rows) >= 25
    assert max(max(r[1:]) for r in rows) <= 1.0, out
