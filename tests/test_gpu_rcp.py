"""The kernels' reciprocal (`fast_rcp`: the hardware seed and one third-order Householder step)
against CUDA's IEEE division, compiled and run as a small program: over 2^24 random mantissas in
every exponent where the operand and its reciprocal are normal, and at the exponents' ends.

Error: the seed is good to 2^-18 or better, the step leaves its cube (below 2^-54) and the rounding
of the last FMA (half a unit), so the result is within one unit of the correctly rounded one."""
import os
import shutil
import subprocess

import pytest

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include <cstdio>
#include "rhi_internal.cuh"
__global__ void worst(long long n, unsigned long long* out) {
    unsigned long long w = 0;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
         i += (long long)gridDim.x * blockDim.x) {
        unsigned long long z = (i + 1) * 0x9E3779B97F4A7C15ULL;
        z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ULL;
        z = (z ^ (z >> 27)) * 0x94D049BB133111EBULL;
        z ^= z >> 31;
        // exponents 2 .. 2044 - 2: the operand and the reciprocal are normal; both signs; all
        // mantissas, and those next to a power of two
        const unsigned long long ex = 2 + (z >> 52) % 2040;
        unsigned long long m = z & 0xFFFFFFFFFFFFFULL;
        if (i % 7 == 0) m &= 3;
        if (i % 7 == 1) m |= 0xFFFFFFFFFFFFCULL;
        const double d = __longlong_as_double((long long)(((z & 1) << 63) | (ex << 52) | m));
        const long long a = __double_as_longlong(rhi::fast_rcp(d)), b = __double_as_longlong(1.0 / d);
        const unsigned long long u = (unsigned long long)(a > b ? a - b : b - a);
        if (u > w) w = u;
    }
    atomicMax(out, w);
}
int main() {
    unsigned long long *d, h = ~0ULL;
    if (cudaMalloc(&d, 8) != cudaSuccess) return 1;
    cudaMemset(d, 0, 8);
    worst<<<304, 256>>>(1LL << 24, d);
    if (cudaMemcpy(&h, d, 8, cudaMemcpyDeviceToHost) != cudaSuccess) return 1;
    printf("%llu\n", h);
    return 0;
}
"""


def test_fast_rcp_is_within_one_unit_of_the_division(tmp_path):
    from paper_0901_1110_gb300 import _build
    src, exe = tmp_path / "rcp.cu", tmp_path / "rcp"
    src.write_text(PROGRAM)
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    subprocess.run([nvcc, *_build.ARCH, "-std=c++17", "-O3", "-I", _build.CSRC, "-I", _build.INCLUDE,
                    "-o", str(exe), str(src)], check=True, capture_output=True, timeout=300)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True, timeout=60)
    assert int(out.stdout) <= 1
