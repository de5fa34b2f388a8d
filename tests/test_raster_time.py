"""The time a raster takes does not depend on how an opening's edges lie in a
cell's height: a thin slot of 4,096 vertices, half of whose edges meet in the
height of one row of cells, against a circle of as many.  They take the same;
three times is the limit (a search that goes round the slot once per edge takes
five to seven times)."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2307_01416_gb300", "csrc")

MAIN = r"""
#include <algorithm>
#include <chrono>
#include <cmath>
#include <cstdio>
#include "tables.h"
using namespace vpmc;
static double fastest(const std::vector<double>& xy)
{
    double best = 1e300;
    for (int k = 0; k < 3; ++k) {
        const auto t = std::chrono::steady_clock::now();
        Raster R{};
        build_raster(xy.data(), (int)(xy.size() / 2), 16.0, &R);
        best = std::min(best, std::chrono::duration<double>(std::chrono::steady_clock::now() - t).count());
    }
    return best;
}
int main()
{
    const int n = 4096;
    std::vector<double> circle, slot;
    for (int i = 0; i < n; ++i) {
        circle.push_back(50.0 * std::cos(2 * M_PI * i / n));
        circle.push_back(50.0 * std::sin(2 * M_PI * i / n));
        const double x = -20.0 + 40.0 * (i % (n / 2)) / (n / 2), ripple = 1e-3 * (i & 1);
        slot.push_back(i < n / 2 ? x : -x);
        slot.push_back((i < n / 2 ? -0.05 : 0.05) + ripple);
    }
    std::printf("%g %g\n", fastest(circle), fastest(slot));
    return 0;
}
"""


def test_a_thin_slot_takes_no_longer_than_a_circle(tmp_path):
    cuda = os.path.join(os.path.dirname(os.path.dirname(shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc")), "include")
    if not shutil.which("g++") or not os.path.exists(os.path.join(cuda, "cuda_runtime.h")):
        pytest.skip("no host compiler or CUDA headers")
    (tmp_path / "main.cpp").write_text(MAIN)
    exe = str(tmp_path / "raster")
    subprocess.run(["g++", "-O3", "-std=c++17", "-pthread", "-I", CSRC, "-I", cuda, str(tmp_path / "main.cpp"),
                    os.path.join(CSRC, "tables.cpp"), "-o", exe], check=True)
    circle, slot = map(float, subprocess.run([exe], check=True, capture_output=True, text=True).stdout.split())
    assert slot <= 3.0 * circle, (circle, slot)
