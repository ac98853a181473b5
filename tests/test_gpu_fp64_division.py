"""The FP64 pair terms' division and reciprocal square root against CUDA's.

The division, bit for bit: its result is the rounded quotient unless the exact one lies within 2^-105 of it of the
middle between two doubles (the error before the last rounding), about one operand pair
in 2^50, so over 2^28 pairs any difference is a fault. The divisor's 2^20 upper
mantissa words are all taken (the hardware's approximation depends on nothing else), with
every exponent from 2^-600 to 2^600 and random lower words; its relative error must stay
below 2^-19, so that the series' truncation e^3 is below 2^-57.

The reciprocal square root: with e = 1 - x y^2 of the approximation below 2^-18, the
step's truncation 5/16 e^3 is below 2^-55.6 and the last rounding 2^-53, so the relative
error stays below 1.17 x 2^-53 (the other roundings enter times e); it is measured from the
residual 1 - x y^2 in two doubles, and CUDA's on the same arguments may not be
smaller by more than a hundredth of a 2^-53.
"""
import os
import subprocess

import pytest

from paper_1904_00861_gb300 import build

pytestmark = pytest.mark.gpu

SRC = r"""
#include <cstdio>
#include "pair64.cuh"
using namespace dtsph;

__device__ unsigned long long mix(unsigned long long z)
{
    z += 0x9E3779B97F4A7C15ull;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}
__device__ double number(unsigned long long bits, int exponent)
{
    return __longlong_as_double((long long)((unsigned long long)(1023 + exponent) << 52 | (bits & 0xfffffffffffffull)));
}
__global__ void check(unsigned long long *bad)
{
    const unsigned long long stride = (unsigned long long)gridDim.x * blockDim.x;
    for (unsigned long long i = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x; i < 1ull << 28; i += stride) {
        const unsigned long long top = i & 0xfffffull, r = mix(i), s = mix(r);
        // 256 rounds over the upper words: exponents in turn and at random, low words at random
        const double b = number(top << 32 | (r & 0xffffffffull), (int)((i >> 20) * 1201 / 256) - 600 + (int)(r >> 63));
        double a = number(s, (int)(mix(s) % 801) - 400);
        if (s >> 63) a = -a;
        if (__double_as_longlong(quotient(a, b)) != __double_as_longlong(a / b)) atomicAdd(&bad[0], 1ull);
        double y;
        asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(b));
        if (!(fabs(__fma_rn(-b, y, 1.0)) < 0x1p-19)) atomicAdd(&bad[1], 1ull);
    }
}
// |1 - y sqrt(x)| of y near 1/sqrt(x): half the residual 1 - x y^2, in two doubles
__device__ double off(double x, double y)
{
    const double yy = y * y, yl = __fma_rn(y, y, -yy), p = x * yy, pl = __fma_rn(x, yy, -p);
    return 0.5 * fabs(((1.0 - p) - pl) - x * yl);
}
__global__ void check_rsqrt(unsigned long long *worst)
{
    const unsigned long long stride = (unsigned long long)gridDim.x * blockDim.x;
    double mine = 0.0, cuda = 0.0, seed = 0.0;
    for (unsigned long long i = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x; i < 1ull << 28; i += stride) {
        const unsigned long long top = i & 0xfffffull, r = mix(i + (1ull << 40));
        const double x = number(top << 32 | (r & 0xffffffffull), (int)((i >> 20) * 1201 / 256) - 600 + (int)(r >> 63));
        mine = fmax(mine, off(x, rsqrt_step(x)));
        cuda = fmax(cuda, off(x, rsqrt(x)));
        double y;
        asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
        seed = fmax(seed, fabs(__fma_rn(-x, y * y, 1.0)));
    }
    atomicMax(&worst[0], (unsigned long long)__double_as_longlong(mine));
    atomicMax(&worst[1], (unsigned long long)__double_as_longlong(cuda));
    atomicMax(&worst[2], (unsigned long long)__double_as_longlong(seed));
}
int main()
{
    unsigned long long *d, h[2] = {1, 1};
    double w[3] = {1, 0, 1};
    cudaMalloc(&d, 5 * 8);
    cudaMemset(d, 0, 5 * 8);
    check<<<608, 256>>>(d);
    check_rsqrt<<<608, 256>>>(d + 2);
    if (cudaMemcpy(h, d, 16, cudaMemcpyDeviceToHost) != cudaSuccess) return 2;
    if (cudaMemcpy(w, d + 2, 24, cudaMemcpyDeviceToHost) != cudaSuccess) return 2;
    printf("%llu quotients differ, %llu seeds are out of bound; rsqrt off by %.4f, CUDA's by %.4f x 2^-53, e %.3g x 2^-18\n",
           h[0], h[1], w[0] * 0x1p53, w[1] * 0x1p53, w[2] * 0x1p18);
    return h[0] || h[1] || !(w[2] < 0x1p-18) || !(w[0] < 1.17 * 0x1p-53) || !(w[0] < w[1] + 0.01 * 0x1p-53);
}
"""


def test_quotient_and_reciprocal_square_root(tmp_path):
    src, exe = tmp_path / "quotient.cu", tmp_path / "quotient"
    src.write_text(SRC)
    subprocess.run([build.nvcc(), *build.ARCH, "-O3", "-std=c++17", "--expt-relaxed-constexpr", "-I" + build.CSRC,
                    "-I" + os.path.join(build.ROOT, "include"), str(src), "-o", str(exe)], check=True,
                   capture_output=True, text=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    print(r.stdout)
    assert r.returncode == 0, r.stdout
