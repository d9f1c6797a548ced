"""The conversions and the division that stand in for FP64 instructions, bit for
bit against those: every float for f2d; for d2f random doubles, and around every
13th float its neighbours' midpoints and the doubles next to them; for div_rn
random pairs, all pairs of edge mantissas and exponents, and quotients next to a
rounding tie. NaN results count as equal whatever their payload."""
import ctypes
import subprocess

import pytest

from paper_2006_16147_gb300 import build

pytestmark = pytest.mark.gpu

SRC = r"""
#include "device_util.cuh"
using namespace amg;
typedef unsigned long long u64;
__device__ u64 mix(u64 x) {                       // splitmix64
    x += 0x9e3779b97f4a7c15ull;
    x = (x ^ (x >> 30)) * 0xbf58476d1ce4e5b9ull;
    x = (x ^ (x >> 27)) * 0x94d049bb133111ebull;
    return x ^ (x >> 31);
}
__device__ double as_d(u64 u) { return __longlong_as_double((long long)u); }
__device__ bool differ(double a, double b) {
    return (a == a || b == b) && __double_as_longlong(a) != __double_as_longlong(b);
}
__device__ bool differ(float a, float b) { return (a == a || b == b) && __float_as_uint(a) != __float_as_uint(b); }
#define EACH(i, n) for (u64 i = blockIdx.x * (u64)blockDim.x + threadIdx.x; i < (n); i += gridDim.x * (u64)blockDim.x)

__global__ void t_f2d(u64* bad) {
    EACH(i, 1ull << 32) {
        const float f = __uint_as_float((unsigned)i);
        if (differ(f2d(f), (double)f)) atomicAdd(bad, 1ull);
    }
}
__global__ void t_d2f(u64* bad, u64 n) {
    EACH(i, n) {
        const u64 r = mix(i);
        const u64 u = i & 1 ? r : (r & ~(0x7ffull << 52)) | ((870 + (r >> 40) % 290) << 52);   // all, or a float's range
        if (differ(d2f(as_d(u)), (float)as_d(u))) atomicAdd(bad, 1ull);
    }
    EACH(i, (1ull << 32) / 13) {
        const float f = __uint_as_float((unsigned)(i * 13)), g = __uint_as_float((unsigned)(i * 13) + 1);
        const u64 mid = (u64)__double_as_longlong(0.5 * ((double)f + (double)g));
        for (int o = -1; o <= 1; ++o)
            if (differ(d2f(as_d(mid + o)), (float)as_d(mid + o))) atomicAdd(bad, 1ull);
    }
}
__device__ u64 edge(unsigned i) {                 // 2 signs x 24 exponents x 24 mantissas
    const u64 es[24] = {0, 1, 2, 3, 52, 53, 54, 970, 1021, 1022, 1023, 1024, 1025, 1075, 1076, 1991, 1992, 2042, 2043,
                        2044, 2045, 2046, 2047, 1000};
    const u64 F = (1ull << 52) - 1;
    const u64 ms[24] = {0, 1, 2, 3, F, F - 1, F - 2, 1ull << 51, (1ull << 51) - 1, (1ull << 51) + 1, 1ull << 29,
                        (1ull << 29) - 1, (1ull << 29) + 1, F ^ ((1ull << 29) - 1), F ^ (1ull << 29), 1ull << 28,
                        0x5555555555555ull, 0xaaaaaaaaaaaaaull, 0x6a09e667f3bcdull, 0x999999999999aull, 1ull << 20,
                        F ^ 0xff, 0x00000fffffffeull, 0xfffff00000001ull};
    return ((u64)(i / 576) << 63) | es[i / 24 % 24] << 52 | ms[i % 24];
}
__global__ void t_div(u64* bad, u64 n) {
    EACH(i, n) {
        const u64 r = mix(2 * i), s = mix(2 * i + 1);
        double a = as_d(r), b = as_d(s);
        if (i % 4) {                              // exponents near 0, so that few pairs leave the integer path
            a = as_d((r & ~(0x7ffull << 52)) | ((1023 - 300 + (r >> 52) % 600) << 52));
            b = as_d((s & ~(0x7ffull << 52)) | ((1023 - 300 + (s >> 52) % 600) << 52));
        }
        if (i % 4 == 2) a = a * b;                // quotient next to a double
        if (i % 4 == 3) {                         // next to a midpoint of two doubles
            const double h = as_d(((u64)__double_as_longlong(a) & (0x7ffull << 52)) - (53ull << 52));
            a = fma(h, b, a * b);
        }
        if (differ(div_rn(a, b), __ddiv_rn(a, b))) atomicAdd(bad, 1ull);
    }
    EACH(i, 1152ull * 1152ull)
        if (differ(div_rn(as_d(edge(i / 1152)), as_d(edge(i % 1152))), __ddiv_rn(as_d(edge(i / 1152)), as_d(edge(i % 1152)))))
            atomicAdd(bad, 1ull);
}
extern "C" int run(int which, u64* bad) {
    u64* d = nullptr;
    if (cudaMalloc(&d, sizeof(u64)) != cudaSuccess) return 1;
    cudaMemset(d, 0, sizeof(u64));
    if (which == 0) t_f2d<<<1024, 256>>>(d);
    if (which == 1) t_d2f<<<1024, 256>>>(d, 1ull << 28);
    if (which == 2) t_div<<<1024, 256>>>(d, 1ull << 28);
    cudaMemcpy(bad, d, sizeof(u64), cudaMemcpyDeviceToHost);
    cudaFree(d);
    return (int)cudaGetLastError();
}
"""


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    at = tmp_path_factory.mktemp("device_math")
    (at / "t.cu").write_text(SRC)
    subprocess.run([build.nvcc(), *build.ARCH, "-O2", "-std=c++17", "-Xcompiler", "-fPIC", "-shared", "-I", build.CSRC,
                    str(at / "t.cu"), "-o", str(at / "t.so")], check=True)
    lib = ctypes.CDLL(str(at / "t.so"))

    def call(which):
        bad = ctypes.c_ulonglong(1)
        assert lib.run(which, ctypes.byref(bad)) == 0
        return bad.value
    return call


@pytest.mark.parametrize("which", ["f2d", "d2f", "div_rn"])
def test_same_bits(run, which):
    assert run(["f2d", "d2f", "div_rn"].index(which)) == 0
