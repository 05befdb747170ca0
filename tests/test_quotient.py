"""quotient.cuh: a quotient from a rounded reciprocal has the bits of the division, on
the host (IEEE) and on the device (CUDA's division): random significands and
exponents, quotients of small integers, zeros, infinities and values at the ends of
fp64's range."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2106_07551_gb300", "csrc")

PROGRAM = r"""
#include <cstdint>
#include <cstdio>
#include <random>
#include <vector>
#include "quotient.cuh"
static bool same(double x, double y) { return (x != x && y != y) || std::memcmp(&x, &y, 8) == 0; }
#ifdef __CUDACC__
__global__ void run(const double* b, const double* a, double* q, double* d, int n) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        q[i] = malib::quotient(b[i], a[i], 1.0 / a[i]);
        d[i] = b[i] / a[i];
    }
}
#endif
int main() {
    std::mt19937_64 r(3);
    std::vector<double> a, b;
    auto wide = [&](int e) { return std::ldexp(1.0 + (double)(r() >> 12) * 0x1p-52, (int)(r() % (2 * e + 1)) - e); };
    for (int i = 0; i < 400000; ++i) {
        a.push_back(wide(i % 4 == 0 ? 1000 : 3));
        b.push_back((i & 1 ? -1 : 1) * wide(i % 8 == 0 ? 1000 : 3));
        a.push_back((double)(1 + r() % 3000));
        b.push_back((double)(r() % 3000));
    }
    for (double x : {0.0, 1.0, 0x1p-1074, 0x1p-1022, 0x1.fffffffffffffp1023, 0x1p500, 0x1p-500, 0x1p-523, (double)INFINITY})
        for (double y : {1.0, 3.0, 1e-12, 0x1p-500, 0x1p499, 0x1p500, 0x1p1023, (double)INFINITY})
            for (double s : {1.0, -1.0}) {
                a.push_back(y);
                b.push_back(s * x);
            }
    const int n = (int)a.size();
    std::vector<double> q(n), d(n);
#ifdef __CUDACC__
    double* m;
    if (cudaMalloc(&m, 4 * sizeof(double) * n) != cudaSuccess) return 2;
    cudaMemcpy(m, b.data(), 8 * n, cudaMemcpyHostToDevice);
    cudaMemcpy(m + n, a.data(), 8 * n, cudaMemcpyHostToDevice);
    run<<<200, 256>>>(m, m + n, m + 2 * n, m + 3 * n, n);
    cudaMemcpy(q.data(), m + 2 * n, 8 * n, cudaMemcpyDeviceToHost);
    if (cudaMemcpy(d.data(), m + 3 * n, 8 * n, cudaMemcpyDeviceToHost) != cudaSuccess) return 2;
#else
    for (int i = 0; i < n; ++i) {
        q[i] = malib::quotient(b[i], a[i], 1.0 / a[i]);
        d[i] = b[i] / a[i];
    }
#endif
    for (int i = 0; i < n; ++i)
        if (!same(q[i], d[i])) { std::printf("%a / %a: %a, not %a\n", b[i], a[i], q[i], d[i]); return 1; }
    return 0;
}
"""


def build_and_run(cmd, tmp_path, name):
    src, exe = tmp_path / name, tmp_path / "quotient"
    src.write_text(PROGRAM)
    subprocess.run([*cmd, "-O2", "-std=c++17", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout


def test_on_the_host(tmp_path):
    build_and_run(["g++", "-ffp-contract=off", "-D__host__=", "-D__device__=", "-D__forceinline__=inline"], tmp_path, "q.cpp")


@pytest.mark.gpu
def test_on_the_device(tmp_path):
    from paper_2106_07551_gb300 import build
    build_and_run([build.nvcc(), *build.ARCH], tmp_path, "q.cu")
