"""The kernels' arithmetic shortcuts against the plain operations, compiled and run as a small program:

- fast_rcp against the division, for every exponent from the smallest normal number to 2^1021 (the range it
  is stated for), 2^27 operands of both signs with random mantissas and those next to a power of two: the
  seed is good to 2^-18 or better, its cube is below 2^-54, and the last FMA rounds by half a unit, so one
  unit at most;
- widen against the conversion, all 2^32 FP32 patterns: exact, NaN for NaN;
- the fast SiLU against the one with a division, all 2^32 patterns: a quotient good to 2^-21 and its residual
  leave 2^-42, under half a unit of rounding each side, so one unit; infinities and NaN alike."""
import os
import shutil
import subprocess

import pytest

pytestmark = pytest.mark.gpu

PROGRAM = r"""
#include <cstdio>
#include "rhi_internal.cuh"
typedef unsigned long long u64;
// units between two numbers by their bit patterns; the zeros count as one number
__device__ u64 dist(long long a, long long b) {
    const long long top = (long long)(1ULL << 63);
    a = a < 0 ? top - a : a;
    b = b < 0 ? top - b : b;
    return (u64)(a > b ? a - b : b - a);
}
__global__ void rcp(long long n, u64* out) {
    u64 w = 0;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        u64 z = (i + 1) * 0x9E3779B97F4A7C15ULL;
        z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ULL;
        z = (z ^ (z >> 27)) * 0x94D049BB133111EBULL;
        z ^= z >> 31;
        const u64 ex = 1 + i % 2043;
        u64 m = z & 0xFFFFFFFFFFFFFULL;
        if (i / 2043 % 7 == 0) m &= 3;
        if (i / 2043 % 7 == 1) m |= 0xFFFFFFFFFFFFCULL;
        const double d = __longlong_as_double((long long)((z >> 63 << 63) | (ex << 52) | m));
        const u64 u = dist(__double_as_longlong(rhi::fast_rcp(d)), __double_as_longlong(1.0 / d));
        if (u > w) w = u;
    }
    atomicMax(out, w);
}
__global__ void wide(u64* out) {
    u64 bad = 0;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < 1LL << 32; i += (long long)gridDim.x * blockDim.x) {
        const float f = __uint_as_float((unsigned)i);
        const double a = rhi::widen(f), b = (double)f;
        if (b != b ? a == a : __double_as_longlong(a) != __double_as_longlong(b)) ++bad;
    }
    if (bad) atomicAdd(out, bad);
}
__global__ void silu(u64* out) {
    u64 w = 0;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < 1LL << 32; i += (long long)gridDim.x * blockDim.x) {
        const float z = __uint_as_float((unsigned)i), a = rhi::silu_f<true>(z), b = rhi::silu_f<false>(z);
        const unsigned ua = __float_as_uint(a), ub = __float_as_uint(b);
        u64 u = dist((long long)((u64)ua << 32), (long long)((u64)ub << 32)) >> 32;
        if (a != a || b != b) u = a != a && b != b ? 0 : 1ULL << 40;
        if (u > w) w = u;
    }
    atomicMax(out, w);
}
int main() {
    u64 *d, h[3] = {~0ULL, ~0ULL, ~0ULL};
    if (cudaMalloc(&d, sizeof h) != cudaSuccess) return 1;
    cudaMemset(d, 0, sizeof h);
    rcp<<<304, 256>>>(1LL << 27, d);
    wide<<<304, 256>>>(d + 1);
    silu<<<304, 256>>>(d + 2);
    if (cudaMemcpy(h, d, sizeof h, cudaMemcpyDeviceToHost) != cudaSuccess) return 1;
    printf("%llu %llu %llu\n", h[0], h[1], h[2]);
    return 0;
}
"""


@pytest.fixture(scope="module")
def worst(tmp_path_factory):
    from paper_0901_1110_gb300 import _build
    tmp = tmp_path_factory.mktemp("arith")
    src, exe = tmp / "arith.cu", tmp / "arith"
    src.write_text(PROGRAM)
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    subprocess.run([nvcc, *_build.ARCH, "-std=c++17", "-O3", "-I", _build.CSRC, "-I", _build.INCLUDE,
                    "-o", str(exe), str(src)], check=True, capture_output=True, timeout=300)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True, timeout=60, env=dict(os.environ))
    return [int(v) for v in out.stdout.split()]


def test_reciprocal_within_one_unit(worst):
    assert worst[0] <= 1, worst


def test_widening_is_exact(worst):
    assert worst[1] == 0, worst


def test_fast_silu_within_one_unit(worst):
    assert worst[2] <= 1, worst
