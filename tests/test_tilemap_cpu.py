"""The tile index of a static launch (csrc/shg_tilemap.cuh) for the longest lists a plan accepts, on the CPU."""
import os
import subprocess

import pytest

from paper_1701_06588_gb300 import build

PROGRAM = r"""
#include "shg_tilemap.cuh"
#include <cstdio>
int main()
{
    // INT32_MAX / 2 pairs, every one with eight lanes
    const int64_t tiles = shg::plan_max_tiles(INT32_MAX / 2, shg::kNClass);
    int64_t bad = tiles > INT32_MAX;
    for (unsigned threads = 32; threads <= 128; threads *= 2) {
        const int64_t per = threads / 32, blocks = (tiles + per - 1) / per;
        for (int64_t b = 0; b < blocks; b += b < 5 || b > blocks - 5 ? 1 : (blocks - 4 - b + 99999) / 100000)
            for (unsigned t = 0; t < threads; ++t)
                bad += shg::launch_warp((unsigned)b, threads, t) != b * per + t / 32;
    }
    std::printf("%lld", (long long)bad);
}
"""


def test_static_launch_covers_the_longest_list(tmp_path):
    try:
        cuda = build._cuda_home()
    except RuntimeError as e:
        pytest.skip(str(e))
    src, exe = tmp_path / "t.cu", tmp_path / "t"
    src.write_text(PROGRAM)
    subprocess.check_call([os.path.join(cuda, "bin", "nvcc"), "-std=c++17", *build.ARCH, "-I" + build.CSRC, "-o", str(exe),
                           str(src)])
    assert subprocess.check_output([str(exe)], text=True) == "0"
