"""The aperture raster's shortcuts against the exact queries, on the CPU: the
host code that builds a raster (csrc/tables.cpp) is compiled into a small
program that asks, for points of every cell near an edge, the crossing-number
test over the cell's local edges and parity, and over all edges, both in FP32
with the kernel's arithmetic.  The answers must agree everywhere (also at a
cell's border, where FP32 placement may pick the neighbouring cell), and the
edge nearest to a cell's centre must never be nearer to a point than the exact
wall distance (it is one of the edges).  Convex, concave, thin and rotated
openings; few and many vertices."""
import os
import shutil
import subprocess

import numpy as np
import pytest

from paper_2307_01416_gb300 import workloads as W

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2307_01416_gb300", "csrc")

MAIN = r"""
#include <cmath>
#include <cstdio>
#include <random>
#include "tables.h"
using namespace vpmc;
int main(int argc, char** argv)
{
    std::FILE* f = std::fopen(argv[1], "rb");
    int n = 0;
    if (!f || std::fread(&n, 4, 1, f) != 1) return 2;
    std::vector<double> xy(2 * n);
    if (std::fread(xy.data(), 8, 2 * n, f) != (size_t)(2 * n)) return 2;
    Raster R{};
    build_raster(xy.data(), n, 16.0, &R);
    std::vector<float> p(2 * n);
    for (int i = 0; i < 2 * n; ++i) p[i] = (float)xy[i];
    auto crosses = [&](float x, float y, int i) {
        const int j = i == 0 ? n - 1 : i - 1;
        const float ax = p[2 * i], ay = p[2 * i + 1], bx = p[2 * j], by = p[2 * j + 1];
        if ((ay > y) == (by > y)) return false;
        return x < ax + (y - ay) * (bx - ax) / (by - ay);
    };
    std::mt19937 g(7);
    std::uniform_real_distribution<float> U(0.0f, 1.0f);
    long asked = 0, listed = 0, cells = 0, wrong = 0;
    for (int cy = 0; cy < kRaster; ++cy)
        for (int cx = 0; cx < kRaster; ++cx) {
            if (R.cells[cy * kRaster + cx] != 2) continue;
            ++cells;
            if (R.near[cy * kRaster + cx] >= n) ++wrong;
            const uint32_t local = R.local[cy * kRaster + cx];
            if (!local) continue;
            ++listed;
            if ((local & 0xffffu) >= (uint32_t)n || ((local >> 16) & 0x7fff) > (uint32_t)kLocalMax) ++wrong;
            for (int k = 0; k < 40; ++k) {
                // inside the cell, on its border, and on a vertex's height
                float u = k < 4 ? (float)(k & 1) : U(g), v = k < 4 ? (float)(k >> 1) : U(g);
                float x = R.lo[0] + (cx + u) / R.inv[0], y = R.lo[1] + (cy + v) / R.inv[1];
                if (k >= 30) {
                    const int i = (int)(local & 0xffffu);
                    const float vy = p[2 * i + 1];
                    if (std::fabs(vy - y) < 1.0f / R.inv[1] && (int)((vy - R.lo[1]) * R.inv[1]) == cy) y = vy;
                }
                bool all = false, loc = (local >> 31) != 0;
                for (int i = 0; i < n; ++i) all ^= crosses(x, y, i);
                int i = (int)(local & 0xffffu);
                for (int c = (int)(local >> 16) & 0x7fff; c > 0; --c) {
                    loc ^= crosses(x, y, i);
                    i = i + 1 < n ? i + 1 : 0;
                }
                ++asked;
                wrong += all != loc;
            }
        }
    std::printf("%ld %ld %ld %ld\n", cells, listed, asked, wrong);
    return 0;
}
"""


def _star(n, r0, r1, turn):
    t = turn + 2 * np.pi * np.arange(n) / n
    r = np.where(np.arange(n) % 2 == 0, r0, r1)
    return np.stack([r * np.cos(t), r * np.sin(t)], axis=1)


def _wavy(n, seed):
    g = np.random.default_rng(seed)
    t = 2 * np.pi * np.arange(n) / n
    r = 12.0 + sum(g.normal(0, 1.5 / k) * np.cos(k * t + g.uniform(0, 6)) for k in range(2, 9))
    return np.stack([r * np.cos(t) + 3.0, r * np.sin(t) - 2.0], axis=1)


POLYGONS = {
    "square": W.square_polygon(6.0),
    "triangle": np.array([[-4.0, -3.0], [5.0, -2.0], [0.5, 7.0]]),
    "slot": np.array([[-20.0, -0.05], [20.0, 0.0], [20.0, 0.1], [-20.0, 0.05]]),
    "comb": np.array([[0, 0], [9, 0], [9, 8], [7, 8], [7, 1], [5, 1], [5, 8], [4, 8], [4, 1], [1, 1], [1, 8], [0, 8.0]]),
    "64-gon": W.regular_polygon(17.6, 64),
    "256-gon": W.regular_polygon(5.0, 256),
    "256-gon turned, clockwise": W.regular_polygon(20.0, 256, center=(4.0, -7.0), phase=0.1)[::-1],
    "star": _star(24, 18.0, 7.0, 0.3),
    "wavy": _wavy(200, 3),
    "many vertices": _wavy(2048, 5),
}


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    cuda = os.path.join(os.path.dirname(os.path.dirname(shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc")), "include")
    if not shutil.which("g++") or not os.path.exists(os.path.join(cuda, "cuda_runtime.h")):
        pytest.skip("no host compiler or CUDA headers")
    d = tmp_path_factory.mktemp("raster")
    (d / "main.cpp").write_text(MAIN)
    exe = str(d / "raster")
    subprocess.run(["g++", "-O2", "-std=c++17", "-pthread", "-ffp-contract=off", "-I", CSRC, "-I", cuda,
                    str(d / "main.cpp"), os.path.join(CSRC, "tables.cpp"), "-o", exe], check=True)
    return exe


@pytest.mark.parametrize("name", list(POLYGONS))
def test_local_edges_decide_as_all_edges(program, name, tmp_path):
    xy = np.ascontiguousarray(POLYGONS[name], dtype=np.float64)
    path = tmp_path / "polygon"
    path.write_bytes(np.int32(len(xy)).tobytes() + xy.tobytes())
    out = subprocess.run([program, str(path)], check=True, capture_output=True, text=True).stdout
    cells, listed, asked, wrong = map(int, out.split())
    assert wrong == 0 and cells > 0 and asked == 40 * listed
    if len(xy) <= 256:                      # ordinary openings: the rule serves nearly every cell
        assert listed >= 0.9 * cells, (cells, listed)
