"""Extended-float arithmetic (csrc/shg_xf.cuh, the same code on host and device) against long double, on the CPU: the
error bounds stated in the header, normalisation, the conversion's range and rounding."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include "shg_xf.cuh"
#include <cmath>
#include <cstdio>
#include <random>
using namespace shg::xfp;
static long double val(xf a) { return std::ldexp((long double)a.m, a.e); }
static bool norm(xf a) { return a.m >= (1ull << 62) && a.m < (1ull << 63); }
int main()
{
    std::mt19937_64 g(1);
    std::uniform_real_distribution<double> u(-60, 60);
    long double em = 0, en = 0, ea = 0, er = 0, ed = 0, ee = 0;
    int bad = 0;
    for (int i = 0; i < 300000; ++i) {
        double x = std::exp2(u(g)), y = std::exp2(u(g));
        if (i % 7 == 0) x = std::ldexp(1.0, (int)(i % 50) - 25);                 // powers of two and their neighbours
        if (i % 11 == 0) x = std::nextafter(x, 0.0);
        const xf a = from_double(x), b = from_double(y), p = mul(a, b), s = add(a, b), q = rsqrt(a);
        const xf n = muln(mulr(a, b), q);
        bad += val(a) != (long double)x || !norm(a) || !norm(p) || !norm(s) || !norm(q) || !norm(n);
        em = std::fmax(em, std::fabs(val(p) / ((long double)x * y) - 1));
        ea = std::fmax(ea, std::fabs(val(s) / ((long double)x + y) - 1));
        er = std::fmax(er, std::fabs(val(q) * std::sqrt((long double)x) - 1));
        en = std::fmax(en, std::fabs(val(n) / (val(q) * x * y) - 1));
        ed = std::fmax(ed, std::fabs(-to_double(p, 0x80000000u) / val(p) - 1));
        const uint64_t Y = g() >> 9;                                             // below 2^55: y <= 2^-9
        ee = std::fmax(ee, std::fabs(std::ldexp((long double)expm1_small(Y), -63) - std::expm1(std::ldexp((long double)Y, -64))));
    }
    bad += to_double(xf{1ull << 62, -2000}, 0) != 0.0 || !std::isinf(to_double(xf{1ull << 62, 2000}, 0));
    bad += to_double(xf{(1ull << 63) - 1, 0}, 0) != 9223372036854775808.0;
    std::printf("%d %.3f %.3f %.3f %.3f %.3f %.3f\n", bad, (double)std::log2(em), (double)std::log2(en), (double)std::log2(ea),
                (double)std::log2(er), (double)std::log2(ed), (double)std::log2(ee));
}
"""


@pytest.mark.skipif(shutil.which("g++") is None, reason="g++ not found")
def test_extended_float_error_bounds(tmp_path):
    src, exe = tmp_path / "xf.cpp", tmp_path / "xf"
    src.write_text(PROGRAM)
    inc = os.path.join(ROOT, "paper_1701_06588_gb300", "csrc")
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-I" + inc, "-o", str(exe), str(src)])
    bad, *err = subprocess.check_output([str(exe)], text=True).split()
    assert int(bad) == 0
    # product, product of a raw product, sum, inverse square root, rounding to FP64, exp(y) - 1 (absolute), in log2
    for e, bound in zip(map(float, err), (-59, -57, -61.9, -58, -52.99, -58)):
        assert e < bound, (err, bound)
