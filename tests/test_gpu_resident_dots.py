"""The dot products of a block of the one-kernel solve: the error of a sum of FP32 terms
does not grow with the rows of the block.  A small CUDA program includes the kernel's source."""
import os
import shutil
import subprocess

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
PKG = os.path.join(ROOT, "paper_1603_04039_gb300")

# Terms all the same are the worst case: the partial sums round the same way for
# long stretches.  1.1771593's squares, 184 in a plain FP32 chain, are off by
# 46 * 2^-24; runs of eight by at most 8 * 2^-24 whatever the terms.
PROGRAM = r"""
#include <cstdio>
#include "resident.cu"

using namespace apc;

__global__ void __launch_bounds__(PB, 1) dots(const float *v, int nv, int R, double *out) {
    __shared__ Fixed S;
    block_dots<float, true>(S, nv, R, [&](int k) -> const float * { return v; }, v, v);
    __syncthreads();
    for (int k = threadIdx.x; k < 2 * nv; k += PB) out[k] = Acc<float>::value(Acc<float>::from(S.val[k]));
}

int main() {
    const int most = PSL * 32;
    const float c = 1.1771593f;
    float *v;
    double *out;
    cudaMallocManaged(&v, most * sizeof(float));
    cudaMallocManaged(&out, RED_SLOTS * sizeof(double));
    for (int r = 0; r < most; ++r) v[r] = c;
    double worst = 0.0;
    int sizes[] = {1, 7, 8, 63, 64, 65, 511, 736, 1472, most}, vectors[] = {2, 3, 5, 24, 25, 32};
    for (int R : sizes)
        for (int nv : vectors) {
            dots<<<1, PB>>>(v, nv, R, out);
            if (cudaDeviceSynchronize() != cudaSuccess) return 2;
            const double want = (double)c * c * R;
            for (int k = 0; k < 2 * nv; ++k) worst = std::max(worst, std::fabs(out[k] - want) / want);
        }
    printf("%.3f\n", worst * 16777216.0);
    return 0;
}
"""


def test_block_sums_do_not_lose_with_the_rows(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not found")
    src, exe = tmp_path / "dots_check.cu", tmp_path / "dots_check"
    src.write_text(PROGRAM)
    subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-O3", "-std=c++17", "-diag-suppress", "550",
                    "-I", os.path.join(PKG, "csrc"), "-I", os.path.join(ROOT, "include"), str(src), "-o", str(exe),
                    "-L", PKG, "-lapcloud", "-Xlinker", "-rpath=" + PKG], check=True, capture_output=True, timeout=300)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True, timeout=120).stdout
    assert float(out) <= 8.0
