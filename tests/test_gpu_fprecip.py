"""FP64 reciprocals and reciprocal square roots from an FP32 start, against exact ones: no
further off than the roundings of their last step allow, over every exponent between 1e-30
and 1e30 and the significands next to powers of two."""
import os
import shutil
import subprocess

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include <cmath>
#include <cstdio>
#include <cstring>
#include <vector>
#include "fprecip.cuh"

__global__ void both(const double *x, double *r, double *q, int n) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    r[i] = apc::recip_f64(x[i]);
    q[i] = apc::rsqrt_f64(x[i]);
}

// |y x - 1| in units of 2^-53: the product and the difference are exact or
// rounded far below that (two fmas)
static double off(double x, double y) { return std::fabs(std::fma(x, y, -1.0)) * 9007199254740992.0; }
// the same for y = 1 / sqrt(x): y^2 x - 1 = 2 d + d^2
static double off_root(double x, double y) {
    const double p = x * y, e = std::fma(x, y, -p);   // x y = p + e
    return 0.5 * std::fabs(std::fma(p, y, -1.0) + e * y) * 9007199254740992.0;
}

int main() {
    std::vector<double> x;
    unsigned long long s = 1;
    for (int e = -99; e < 100; ++e) {
        for (int k = 0; k < 5000; ++k) {
            s = s * 6364136223846793005ull + 1442695040888963407ull;
            x.push_back(std::ldexp(1.0 + (double)(s >> 12) * std::ldexp(1.0, -52), e));
        }
        for (int k = 0; k < 64; ++k) {
            x.push_back(std::ldexp(1.0 + k * std::ldexp(1.0, -52), e));
            x.push_back(std::ldexp(2.0 - (k + 1) * std::ldexp(1.0, -52), e));
        }
    }
    const int n = (int)x.size();
    double *gx, *gr, *gq;
    cudaMalloc(&gx, n * 8); cudaMalloc(&gr, n * 8); cudaMalloc(&gq, n * 8);
    cudaMemcpy(gx, x.data(), n * 8, cudaMemcpyHostToDevice);
    both<<<(n + 255) / 256, 256>>>(gx, gr, gq, n);
    if (cudaDeviceSynchronize() != cudaSuccess) return 2;
    std::vector<double> r(n), q(n);
    cudaMemcpy(r.data(), gr, n * 8, cudaMemcpyDeviceToHost);
    cudaMemcpy(q.data(), gq, n * 8, cudaMemcpyDeviceToHost);
    double a = 0, b = 0;
    for (int i = 0; i < n; ++i) {
        a = std::fmax(a, off(x[i], r[i]));
        b = std::fmax(b, off_root(x[i], q[i]));
    }
    printf("n %d recip %.6f rsqrt %.6f\n", n, a, b);
    return 0;
}
"""


def test_reciprocals(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not found")
    src, exe = tmp_path / "recip_check.cu", tmp_path / "recip_check"
    src.write_text(PROGRAM)
    subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-O3", "-std=c++17", "-Xcompiler", "-ffp-contract=off",
                    "-I", os.path.join(ROOT, "paper_1603_04039_gb300", "csrc"), str(src), "-o", str(exe)],
                   check=True, capture_output=True, timeout=300)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True, timeout=120).stdout.split()
    assert int(out[1]) > 900_000
    # relative to 1: a last rounding of at most 2^-53; the root's product g y adds half of that
    assert float(out[3]) <= 1.0 + 1e-3 and float(out[5]) <= 1.5 + 1e-2
