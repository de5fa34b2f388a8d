"""Failed waits of the surrogate's tensor-core kernels.  surrogate.cu is
compiled with a small program whose fake of the wait's result lets one thread
of the first block see one of its waits fail.  The fake waits like the real one
first, so the work is complete and nothing hangs or faults; what is tested is
what the kernel does with the answer.  The program prints the status word, that
thread's waits (barrier and parity, in order) and which outputs were written.
A whole tile of the forward kernel waits for its inputs and then for three
GEMMs, a ragged one for the GEMMs alone."""
import os
import shutil
import subprocess

import pytest

from paper_2307_01416_gb300 import build_ext

pytestmark = pytest.mark.gpu

MAIN = r"""
#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include <vector>
__device__ int fake_thread, fake_call, fake_n;
__device__ unsigned fake_log[256][2];
__device__ bool fake_result(uint32_t mbar, uint32_t parity, bool done)
{
    if (blockIdx.x != 0 || (int)threadIdx.x != fake_thread) return done;
    const int i = fake_n++;
    if (i < 256) { fake_log[i][0] = mbar; fake_log[i][1] = parity; }
    return done && i != fake_call;
}
#define VPMC_WAIT_RESULT(mbar, parity, done) fake_result(mbar, parity, done)
#include "surrogate.cu"

using namespace vpmc;
template <class T> T* device(size_t n)
{
    T* p = nullptr;
    if (cudaMalloc(&p, n * sizeof(T)) != cudaSuccess || cudaMemset(p, 0, n * sizeof(T)) != cudaSuccess) std::exit(3);
    return p;
}
int main(int, char** argv)      // forward | train, rows, thread, call
{
    const bool train = argv[1][0] == 't';
    const long long n = std::atoll(argv[2]);
    const int thread = std::atoi(argv[3]), call = std::atoi(argv[4]);
    SurNet net{};
    net.params = device<float>(sur::kNParams);
    net.gpart = device<float>(sur::kNParams);
    net.n_part_cap = 1;
    net.img = device<unsigned char>(sur::kImgBytes);
    net.loss = device<double>(2);
    net.status = device<int>(1);
    std::vector<float> w(sur::kNParams), x(6 * n), y(5 * n, 0.25f), z(45 * n, -1e30f), g(sur::kNParams);
    std::vector<int> label(n, 1);
    uint32_t seed = 1;
    auto uniform = [&] { seed = seed * 1664525u + 1013904223u; return (float)(seed >> 8) * 0x1p-23f - 1.0f; };
    for (float& v : w) v = 0.1f * uniform();
    for (float& v : x) v = uniform();
    float *dx = device<float>(x.size()), *dy = device<float>(y.size()), *dz = device<float>(z.size());
    int* dl = device<int>(n);
    cudaMemcpy(net.params, w.data(), 4 * w.size(), cudaMemcpyHostToDevice);
    cudaMemcpy(dx, x.data(), 4 * x.size(), cudaMemcpyHostToDevice);
    cudaMemcpy(dy, y.data(), 4 * y.size(), cudaMemcpyHostToDevice);
    cudaMemcpy(dz, z.data(), 4 * z.size(), cudaMemcpyHostToDevice);
    cudaMemcpy(dl, label.data(), 4 * n, cudaMemcpyHostToDevice);
    cudaMemcpyToSymbol(fake_thread, &thread, 4);
    cudaMemcpyToSymbol(fake_call, &call, 4);
    int parts = 0, status = 0, calls = 0;
    cudaError_t e = launch_sur_pack(net, 0);
    if (e == cudaSuccess)
        e = train ? launch_sur_train(net, dx, dy, dl, 0, n, n, 1.0f / n, 1, &parts, 0) : launch_sur_forward(net, dx, n, dz, 1, 0);
    if (e == cudaSuccess) e = cudaDeviceSynchronize();
    if (e != cudaSuccess) { std::printf("%s\n", cudaGetErrorString(e)); return 4; }
    cudaMemcpy(&status, net.status, 4, cudaMemcpyDeviceToHost);
    cudaMemcpyFromSymbol(&calls, fake_n, 4);
    unsigned log[256][2];
    cudaMemcpyFromSymbol(log, fake_log, sizeof log);
    cudaMemcpy(z.data(), dz, 4 * z.size(), cudaMemcpyDeviceToHost);
    cudaMemcpy(g.data(), net.gpart, 4 * g.size(), cudaMemcpyDeviceToHost);
    std::printf("status %d\nwaits", status);
    for (int i = 0; i < calls && i < 256; ++i) std::printf(" %u:%u", log[i][0], log[i][1]);
    std::printf("\ntiles");                     // written values per tile of 128 rows
    for (long long t = 0; t < (n + 127) / 128; ++t) {
        int k = 0;
        for (long long i = 45 * 128 * t; i < 45 * 128 * (t + 1) && i < 45 * n; ++i) k += z[i] != -1e30f;
        std::printf(" %d", k);
    }
    int k = 0;
    for (float v : g) k += v != 0.0f;
    std::printf("\ngradient %d\n", k);
    return 0;
}
"""


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    if not (shutil.which("nvcc") or os.path.exists("/usr/local/cuda/bin/nvcc")):
        pytest.skip("no nvcc")
    d = tmp_path_factory.mktemp("waits")
    (d / "main.cu").write_text(MAIN)
    exe = str(d / "waits")
    subprocess.run([build_ext._nvcc()] + build_ext.ARCH + build_ext.NVCC_FLAGS + [str(d / "main.cu"), "-o", exe], check=True)

    def call(kind, rows, thread, call):
        out = subprocess.run([exe, kind, str(rows), str(thread), str(call)], check=True, capture_output=True, text=True,
                             timeout=120).stdout
        r = {k: v.split() for k, v in (line.split(" ", 1) for line in out.strip().splitlines() if " " in line)}
        return {"status": int(r["status"][0]), "waits": [tuple(map(int, w.split(":"))) for w in r.get("waits", [])],
                "tiles": list(map(int, r["tiles"])), "gradient": int(r["gradient"][0])}

    return call


@pytest.mark.parametrize("rows,first", [(128, 1), (100, 0)], ids=["whole tile", "ragged tile"])
@pytest.mark.parametrize("thread", [0, 1, 77, 127])
def test_forward_stops_at_a_failed_wait(run, rows, first, thread):
    """Whichever thread's wait for a GEMM fails: the call reports it, the tile
    is not stored, no further GEMM is waited for, and the phase that was open is
    waited for once more before the tensor memory is given back."""
    clean = run("forward", rows, thread, -1)
    assert clean["status"] == 0 and clean["tiles"] == [45 * rows] and len(clean["waits"]) == first + 3
    for gemm in range(3):
        r = run("forward", rows, thread, first + gemm)
        assert r["status"] == 1 and r["tiles"] == [0]
        assert r["waits"] == clean["waits"][:first + gemm + 1] + [clean["waits"][first + gemm]]


def test_other_pipelines_and_earlier_tiles_are_unaffected(run):
    """Ten tiles on one block's four pipelines: the second tile of pipeline 0
    fails, so that its third one is not begun; the others are whole."""
    r = run("forward", 10 * 128, 77, 4 + 2)
    assert r["status"] == 1
    assert r["tiles"] == [0 if t in (4, 8) else 45 * 128 for t in range(10)]


@pytest.mark.parametrize("thread", [0, 77, 511])
def test_training_stops_at_a_failed_wait(run, thread):
    """Two tiles of one block: the weight images, then six GEMM phases a tile.
    A failed phase is reported, ends the block's work, leaves its partial
    gradient at zero and is waited for once more."""
    clean = run("train", 256, thread, -1)
    assert clean["status"] == 0 and clean["gradient"] > 0 and len(clean["waits"]) == 13
    for call in range(1, 13):
        r = run("train", 256, thread, call)
        assert r["status"] == 1 and r["gradient"] == 0
        assert r["waits"] == clean["waits"][:call + 1] + [clean["waits"][call]]


@pytest.mark.parametrize("thread", [0, 77, 127])
def test_copies_in_flight_are_waited_for(run, thread):
    """A bulk copy whose wait failed, or that was started for a tile that is
    not begun any more, is waited for once more; no GEMM is begun without it."""
    clean = run("forward", 128, thread, -1)
    r = run("forward", 128, thread, 0)
    assert r["status"] == 1 and r["tiles"] == [0] and r["waits"] == 2 * clean["waits"][:1]
    # the first GEMM fails while the pipeline's next inputs are on their way
    r = run("forward", 10 * 128, thread, 1)
    inputs, gemm = clean["waits"][:2]
    assert r["status"] == 1 and r["tiles"] == [0 if t % 4 == 0 else 45 * 128 for t in range(10)]
    assert r["waits"][:2] == [inputs, gemm] and sorted(r["waits"][2:]) == sorted([(inputs[0], 1 - inputs[1]), gemm])
    clean = run("train", 256, thread, -1)
    r = run("train", 256, thread, 0)
    assert r["status"] == 1 and r["gradient"] == 0 and r["waits"] == 2 * clean["waits"][:1]
