"""The generator's per-history prepared words against the plain ten rounds, on
the CPU: the device header's two functions are compiled for the host and
compared over keys, histories and steps with extreme words among them."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2307_01416_gb300", "csrc")

MAIN = r"""
#include <cstdio>
#include "device_common.cuh"
using namespace vpmc::dev;

template <class F> int over(F f)
{
    const uint32_t w[] = {0u, 1u, 2u, 31u, 0x7fffffffu, 0x80000000u, 0xfffffffeu, 0xffffffffu, 0x9E3779B9u, 0xBB67AE85u,
                          1234u, 0xCD9E8D57u};
    int wrong = 0;
    for (uint32_t a : w) for (uint32_t b : w) for (uint32_t h : w) for (uint32_t s : w) wrong += f(a, b, h, s);
    return wrong;
}
int main()
{
    const int wrong = over([](uint32_t a, uint32_t b, uint32_t h, uint32_t s) {
        const uint2 k = make_uint2(a, b);
        const uint4 p = philox(make_uint4(h, s, 1u, 0u), k), q = philox_step(s, k, philox_step_prepare(h, k));
        return p.x != q.x || p.y != q.y || p.z != q.z || p.w != q.w;
    });
    std::printf("%d\n", wrong);
    return wrong != 0;
}
"""


def test_prepared_words_give_the_same_block(tmp_path):
    if not shutil.which("nvcc"):
        pytest.skip("no nvcc")
    src = tmp_path / "main.cu"
    src.write_text(MAIN)
    header = tmp_path / "host"
    header.mkdir()
    # the functions under test, as host functions
    for name in ("device_common.cuh", "vpmc_internal.cuh"):
        text = open(os.path.join(CSRC, name)).read()
        if name == "device_common.cuh":
            text = text[:text.index("// ((x >> 9) + 1/2)")].replace("__device__ __forceinline__", "inline") + "}\n}\n"
        (header / name).write_text(text)
    exe = str(tmp_path / "philox")
    subprocess.run(["nvcc", "-std=c++17", "-O1", "-I", str(header), str(src), "-o", exe], check=True)
    assert subprocess.run([exe], capture_output=True, text=True).stdout.strip() == "0"
