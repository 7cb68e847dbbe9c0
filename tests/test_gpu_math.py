"""The step's and the surrogate's own elementary functions against CUDA's, through a small library
compiled here from the same headers."""
import ctypes
import os
import subprocess

import pytest

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include "lbm_kernels.cuh"
#include "step64.cuh"
namespace {  // what mlp_infer.cuh takes from the network's layout
constexpr int kIn = 4, kHid = 128, kOut = 4;
__host__ __device__ constexpr int woff(int) { return 0; }
[[maybe_unused]] __host__ __device__ constexpr int boff(int) { return 0; }
}
#include "mlp_infer.cuh"

__device__ unsigned long long g_bad[2];
__device__ double g_max[4];

__device__ void at_most(double* slot, double v) {  // v >= 0 (NaN counts as infinite)
    atomicMax(reinterpret_cast<unsigned long long*>(slot), (unsigned long long)__double_as_longlong(isnan(v) ? INFINITY : v));
}
__device__ double ulps(double got, double want) {
    return (double)llabs(__double_as_longlong(got) - __double_as_longlong(want));
}
__device__ unsigned long long mix(unsigned long long z) {  // SplitMix64 (Steele, Lea and Flood 2014)
    z = (z + 0x9e3779b97f4a7c15ull);
    z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ull;
    z = (z ^ (z >> 27)) * 0x94d049bb133111ebull;
    return z ^ (z >> 31);
}
// a double of exponent lo .. hi (inclusive) and random significand, some at its ends
__device__ double argument(unsigned long long i, int lo, int hi) {
    const unsigned long long r = mix(i);
    const int e = lo + (int)((r >> 52) % (unsigned)(hi - lo + 1));
    unsigned long long m = r & 0xfffffffffffffull;
    if (i % 64 == 0) m = (i >> 6) % 4096;
    if (i % 64 == 1) m = 0xfffffffffffffull - (i >> 6) % 4096;
    return __longlong_as_double(((long long)(e + 1023) << 52) | (long long)m);
}

// every significand of exponent e, one cell and the two cells of a pair
__global__ void fp32(int e) {
    for (unsigned m = blockIdx.x * blockDim.x + threadIdx.x; m < 1u << 23; m += gridDim.x * blockDim.x) {
        const float x = __uint_as_float((unsigned)(e + 127) << 23 | m), y = __uint_as_float((unsigned)(e + 127) << 23 | (m ^ 0x2aaaaa));
        const lbmk::F2 r = lbmk::rcp_v(lbmk::F2(x, y)), s = lbmk::sqrt_v(lbmk::F2(x, y));
        if (r.v.x != __frcp_rn(x) || r.v.y != __frcp_rn(y) || lbmk::rcp_v(lbmk::F1(x)).v != __frcp_rn(x)) atomicAdd(&g_bad[0], 1ull);
        if (s.v.x != __fsqrt_rn(x) || s.v.y != __fsqrt_rn(y) || lbmk::sqrt_v(lbmk::F1(x)).v != __fsqrt_rn(x)) atomicAdd(&g_bad[1], 1ull);
    }
}
__global__ void fp64(long long n) {
    double a = 0, b = 0;
    unsigned long long na = 0, nb = 0;
    for (long long i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const double x = argument(i, -40, 40);
        const double u = ulps(lbmk::rcp_d(x), 1.0 / x), v = ulps(lbmk::sqrt_d(x), sqrt(x));
        a = fmax(a, u), b = fmax(b, v), na += u != 0, nb += v != 0;
    }
    at_most(&g_max[0], a), at_most(&g_max[1], b);
    atomicAdd(&g_bad[0], na), atomicAdd(&g_bad[1], nb);
}
// largest |error| in units of 1.5 ulp of ln x + 2.2e-17
__global__ void logarithm(long long n) {
    lbmk::LogTable t;
    t.load();
    double a = 0;
    for (long long j = blockIdx.x * (blockDim.x / 32) + threadIdx.x / 32; j < n / 32; j += gridDim.x * (blockDim.x / 32)) {
        const long long i = 32 * j + threadIdx.x % 32;
        const double x = argument(i, i % 2 ? -1 : -20, i % 2 ? 0 : 6), l = log(x);
        const double ulp = l == 0.0 ? 0.0 : __longlong_as_double(__double_as_longlong(fabs(l)) + 1) - fabs(l);
        a = fmax(a, fabs(lbmk::log_d(x, t) - l) / (1.5 * ulp + 2.2e-17));
    }
    at_most(&g_max[2], a);
}
// largest |error| of gelu2, one in 16 of all finite z, in units of 2^-23.5 + 2^-24 |gelu|
__global__ void gelu() {
    double a = 0;
    for (unsigned i = blockIdx.x * blockDim.x + threadIdx.x; i < 0x7f80000u; i += gridDim.x * blockDim.x) {
        const float z = __uint_as_float(16 * i + (i * 7 & 15));
        const float2 g = gelu2(make_float2(z, -z));
        for (int k = 0; k < 2; ++k) {
            const double x = k ? -z : z, want = 0.5 * x * erfc(-x * 0.70710678118654752440), got = k ? g.y : g.x;
            a = fmax(a, fabs(got - want) / (8.4293697021788057e-08 + 5.9604644775390625e-08 * fabs(want)));
        }
    }
    at_most(&g_max[3], a);
}

extern "C" int math_check(unsigned long long* bad, double* max4) {
    unsigned long long b[2], z[2] = {0, 0};
    const double zm[4] = {0, 0, 0, 0};
    cudaMemcpyToSymbol(g_bad, z, sizeof(z));
    cudaMemcpyToSymbol(g_max, zm, sizeof(zm));
    for (int e = -40; e <= 40; ++e) fp32<<<608, 256>>>(e);
    cudaMemcpyFromSymbol(b, g_bad, sizeof(b));
    bad[0] = b[0], bad[1] = b[1];
    cudaMemcpyToSymbol(g_bad, z, sizeof(z));
    fp64<<<608, 256>>>(1 << 24);
    logarithm<<<608, 256>>>(1 << 24);
    gelu<<<608, 256>>>();
    cudaMemcpyFromSymbol(bad + 2, g_bad, sizeof(b));
    cudaMemcpyFromSymbol(max4, g_max, sizeof(zm));
    return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def checked(tmp_path_factory):
    import torch

    from paper_2403_11167_gb300 import build

    assert torch.cuda.is_available()
    d = tmp_path_factory.mktemp("math")
    src, so = d / "check.cu", d / "check.so"
    src.write_text(SOURCE)
    subprocess.run([build.NVCC, *build.ARCH, "-O3", "-std=c++17", "-shared", "-Xcompiler", "-fPIC", "-I", build.CSRC,
                    str(src), "-o", str(so)], check=True)
    lib = ctypes.CDLL(str(so), mode=os.RTLD_LOCAL)
    bad, mx = (ctypes.c_ulonglong * 4)(), (ctypes.c_double * 4)()
    assert lib.math_check(bad, mx) == 0
    return list(bad), list(mx)


def test_fp32_reciprocal_and_root_are_correctly_rounded(checked):
    """Every significand of exponents -40 .. 40: the bits of __frcp_rn and __fsqrt_rn."""
    assert checked[0][:2] == [0, 0]


def test_fp64_reciprocal_and_root(checked):
    """Exponents -40 .. 40.  An approximation of 20 bits and one cubic step leave 2^-60 of the reciprocal before
    its last rounding, 2^-7 ulp: at most an ulp off, and in few cases (a 50th at most).  The root's last step
    corrects an error of 2^-39 to 2^-78: rounded correctly but where that is a tie, one in a million at most."""
    bad, mx = checked
    print("FP64 reciprocal, root: not correctly rounded", bad[2:], "of", 1 << 24, "largest", mx[:2])
    assert mx[0] <= 1 and bad[2] <= (1 << 24) / 50
    assert mx[1] <= 1 and bad[3] <= (1 << 24) / 1e6


def test_fp64_logarithm(checked):
    """Arguments of 2^-20 .. 2^6 and around 1: within 1.5 ulp and 2.2e-17 of CUDA's log (an ulp is log's own and half
    of one the last sum's; the table's values are good to 6e-18, the polynomial to 1.3e-17, and three numbers
    below 1/64 are rounded by 2^-60 each)."""
    assert checked[1][2] <= 1.0, checked[1][2]


def test_gelu(checked):
    """All finite z: within 2^-23.5 and 2^-24 of the value of z Phi(z) in 64 bits (ex2.approx 2^-22 and the exponent's
    roundings 3 x 2^-24 of at most 0.17, the polynomial, and the last rounding)."""
    assert checked[1][3] <= 1.0, checked[1][3]
