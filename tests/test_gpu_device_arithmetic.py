"""The conversions between 32 and 64 bits by integer operations and the double
reciprocal, against the instructions they stand for: every float, doubles over
the whole exponent range with its ends, values next to ties."""
import os
import subprocess

import pytest

from paper_1507_02509_gb300 import build as kbuild

pytestmark = pytest.mark.gpu

PROGRAM = r"""
#include <cstdio>
#include <cuda_fp16.h>
#include "kbc_lattice.cuh"

using namespace kbc;

__device__ unsigned long long mix(unsigned long long x)
{
    x += 0x9e3779b97f4a7c15ull;
    x = (x ^ (x >> 30)) * 0xbf58476d1ce4e5b9ull;
    x = (x ^ (x >> 27)) * 0x94d049bb133111ebull;
    return x ^ (x >> 31);
}
// any bits; or one of: few low bits set, a float's tie, a half's tie, all ones
__device__ double pattern(unsigned long long k)
{
    const unsigned long long a = mix(2 * k), b = mix(2 * k + 1), top = a & 0xfff0000000000000ull;
    unsigned long long f = b & 0x000fffffffffffffull;
    switch (k & 7) {
    case 1: f = f & ~((1ull << (k >> 3 & 63) % 53) - 1) & 0x000fffffffffffffull; break;
    case 2: f = (f & ~0x1fffffffull) | 0x10000000ull; break;
    case 3: f = ((f & ~0x1fffffffull) | 0x10000000ull) + (b >> 60) - 8; break;
    case 4: f = (f & ~0x3ffffffffffull) | 0x20000000000ull; break;
    case 5: f = ((f & ~0x3ffffffffffull) | 0x20000000000ull) + (b >> 60) - 8; break;
    case 6: f = 0x000fffffffffffffull - (b >> 58); break;
    case 7: f = b >> 58; break;
    }
    unsigned long long v = top | (f & 0x000fffffffffffffull);
    // exponents around those of float and half in half of the cases
    if (k & 8) v = (v & 0x800fffffffffffffull) | ((unsigned long long)(860 + (a >> 3) % 330) << 52);
    return __longlong_as_double((long long)v);
}
__device__ bool same(double a, double b)
{
    return __double_as_longlong(a) == __double_as_longlong(b) || (isnan(a) && isnan(b));
}
__device__ bool same(float a, float b)
{
    return __float_as_uint(a) == __float_as_uint(b) || (isnan(a) && isnan(b));
}

// out: wrong widen, narrow, narrow_odd, special reciprocals; reciprocals one
// unit off, further off, compared
__global__ void compare(unsigned long long* out, unsigned long long doubles)
{
    unsigned long long bad[7] = {0, 0, 0, 0, 0, 0, 0};
    const unsigned long long t = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x;
    const unsigned long long threads = (unsigned long long)gridDim.x * blockDim.x;
    for (unsigned long long k = t; k < (1ull << 32); k += threads) {
        const float v = __uint_as_float((unsigned)k);
        bad[0] += !same(widen(v), (double)v);
    }
    for (unsigned long long k = t; k < doubles; k += threads) {
        const double v = pattern(k);
        bad[1] += !same(narrow(v), __double2float_rn(v));
        const __half a = __float2half_rn(narrow_odd(v)), b = __double2half(v);
        bad[2] += __half_as_ushort(a) != __half_as_ushort(b) && !(__hisnan(a) && __hisnan(b));
        const double q = 1.0 / v, r = rcp_pos(v);
        const long long x = llabs(__double_as_longlong(v));
        if (__double_as_longlong(v) <= 0 || x < 0x0010000000000000ll || x >= 0x7fd0000000000000ll) {
            bad[3] += !same(q, r);  // not a positive normal with a normal reciprocal
        } else {
            const long long d = llabs(__double_as_longlong(q) - __double_as_longlong(r));
            bad[4] += d == 1;
            bad[5] += d > 1;
            ++bad[6];
        }
    }
    for (int j = 0; j < 7; ++j)
        if (bad[j]) atomicAdd(out + j, bad[j]);
}

int main()
{
    unsigned long long *out, h[7];
    if (cudaMalloc(&out, sizeof h) || cudaMemset(out, 0, sizeof h)) return 2;
    compare<<<152 * 8, 256>>>(out, 1ull << 26);
    if (cudaMemcpy(h, out, sizeof h, cudaMemcpyDeviceToHost)) return 3;
    for (int j = 0; j < 7; ++j) std::printf("%llu ", h[j]);
    return 0;
}
"""


def test_conversions_and_reciprocals(tmp_path):
    src = tmp_path / "arith.cu"
    src.write_text(PROGRAM)
    exe = tmp_path / "arith"
    subprocess.run([kbuild.nvcc(), *kbuild.ARCH, "-O3", "-std=c++17", "--expt-relaxed-constexpr", "-I", kbuild.CSRC,
                    str(src), "-o", str(exe)], check=True, env={**os.environ})
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout + r.stderr
    widen, narrow, odd, special, one_off, further, compared = map(int, r.stdout.split())
    assert (widen, narrow, odd, special, further) == (0, 0, 0, 0, 0)
    # the remainder of the series is 2^-20 of the last bit: that part of the values, twice
    assert compared > 1 << 24 and one_off <= compared * 2.0 ** -19
