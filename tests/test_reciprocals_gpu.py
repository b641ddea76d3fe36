"""The branch-free reciprocals of the kernels against CUDA's division, compiled from the kernels' own sources: every
float whose reciprocal is normal, every argument of the logistic function, and a spread of doubles."""
import ctypes
import subprocess

import pytest
import torch

from paper_2409_01076_gb300 import build_lib

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include "nn_vec.cu"
#include "d2q9.cuh"

using u64 = unsigned long long;

// Counts x with exponents 2^-126 to 2^125, either sign, where r(x) is not 1 / x to the bit.
__global__ void floats(u64 *bad)
{
    u64 n = 0;
    for (u64 k = blockIdx.x * (u64)blockDim.x + threadIdx.x; k < (1ull << 32); k += (u64)gridDim.x * blockDim.x) {
        const unsigned b = (unsigned)k, e = (b >> 23) & 255u;
        if (e < 1 || e > 252) continue;
        const float x = __uint_as_float(b);
        const smrt::F2 one = smrt::f2(1.0f, 1.0f), r = smrt::vrecip_neg(smrt::f2(-x, -x), one);
        const unsigned want = __float_as_uint(1.0f / x);
        n += __float_as_uint(smrt::f2_lo(r)) != want || __float_as_uint(smrt::f2_hi(r)) != want;
    }
    atomicAdd(bad, n);
}

// Counts z where the logistic function is not the rounded quotient.
__global__ void logistic(u64 *bad)
{
    u64 n = 0;
    for (u64 k = blockIdx.x * (u64)blockDim.x + threadIdx.x; k < (1ull << 32); k += (u64)gridDim.x * blockDim.x) {
        const float z = __uint_as_float((unsigned)k);
        if (z != z) { n += sigm(z) == sigm(z); continue; }
        n += __float_as_uint(sigm(z)) != __float_as_uint(1.0f / (1.0f + expf(-z)));
    }
    atomicAdd(bad, n);
}

// Doubles of 2,045 exponents, mantissas by a multiplicative sequence: those more than one unit in the last place off.
__global__ void doubles(u64 count, u64 *bad)
{
    u64 n = 0;
    for (u64 k = blockIdx.x * (u64)blockDim.x + threadIdx.x; k < count; k += (u64)gridDim.x * blockDim.x) {
        const u64 h = (k + 1) * 0x9E3779B97F4A7C15ull, e = 1 + k % 2044;
        const double x = __longlong_as_double((long long)((h & 0x800FFFFFFFFFFFFFull) | (e << 52)));
        const long long d = __double_as_longlong(smrt::recip_d(x)) - __double_as_longlong(1.0 / x);
        n += d < -1 || d > 1;
    }
    atomicAdd(bad, n);
}

extern "C" __attribute__((visibility("default"))) int run(int which, u64 count, u64 *bad)
{
    if (which == 0) floats<<<1216, 256>>>(bad);
    else if (which == 1) logistic<<<1216, 256>>>(bad);
    else doubles<<<1216, 256>>>(count, bad);
    const cudaError_t e = cudaGetLastError();
    return (int)(e != cudaSuccess ? e : cudaDeviceSynchronize());
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("reciprocals")
    src, so = d / "reciprocals.cu", d / "reciprocals.so"
    src.write_text(SOURCE)
    subprocess.run([build_lib.nvcc(), *build_lib.ARCH, *build_lib.NVCC_FLAGS, "-shared", str(src), "-o", str(so)],
                   check=True, capture_output=True, text=True)
    torch.cuda.init()
    lib = ctypes.CDLL(str(so))
    lib.run.argtypes = [ctypes.c_int, ctypes.c_ulonglong, ctypes.c_void_p]
    return lib


@pytest.mark.parametrize("which,count", [(0, 0), (1, 0), (2, 200_000_000)], ids=["float", "logistic", "double"])
def test_equal_to_the_division(lib, which, count):
    bad = torch.zeros(1, dtype=torch.int64, device="cuda")
    torch.cuda.synchronize()
    assert lib.run(which, count, bad.data_ptr()) == 0
    assert int(bad.item()) == 0
