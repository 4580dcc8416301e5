"""The conversion of extended floats (csrc/shg_xf.cuh) at the ends of the FP64 range: every normal value comes back exactly,
the largest binade included, and what rounds beyond it is infinite."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include "shg_xf.cuh"
#include <cfloat>
#include <initializer_list>
#include <cmath>
#include <cstdio>
using namespace shg::xfp;
int main()
{
    int bad = 0;
    for (int e = -1022; e <= 1023; ++e)
        for (double f : {1.0, 1.0 + DBL_EPSILON, 1.5, 2.0 - DBL_EPSILON}) {
            const double x = std::ldexp(f, e);
            bad += to_double(from_double(x), 0) != x || to_double(from_double(x), 0x80000000u) != -x;
        }
    // half an ulp above the largest value rounds up, less does not
    const xf top = from_double(DBL_MAX);
    bad += to_double(xf{top.m + 511, top.e}, 0) != DBL_MAX || !std::isinf(to_double(xf{top.m + 512, top.e}, 0));
    for (int e = top.e + 1; e < top.e + 5000; ++e) bad += !std::isinf(to_double(xf{1ull << 62, e}, 0));
    const xf least = from_double(DBL_MIN);
    for (int e = least.e - 1; e > least.e - 5000; --e) bad += to_double(xf{1ull << 62, e}, 0) != 0.0;
    std::printf("%d", bad);
}
"""


@pytest.mark.skipif(shutil.which("g++") is None, reason="g++ not found")
def test_conversion_over_the_whole_range(tmp_path):
    src, exe = tmp_path / "r.cpp", tmp_path / "r"
    src.write_text(PROGRAM)
    inc = os.path.join(ROOT, "paper_1701_06588_gb300", "csrc")
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-I" + inc, "-o", str(exe), str(src)])
    assert subprocess.check_output([str(exe)], text=True) == "0"
