"""The quotients of the single-precision D (reciprocal_rn, quotient_rn and D_of_f of
fld_device.cuh) against the correctly rounded operations, bit for bit: the
reciprocal for every mantissa, D over its whole range and at the ends where it
changes its way.  The device code is compiled with a small kernel of the test."""
import ctypes
import os
import subprocess

import pytest

pytestmark = pytest.mark.gpu

fld = pytest.importorskip("paper_1403_8105_gb300")
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_1403_8105_gb300 import _build  # noqa: E402

_CODE = r"""
#include <cuda_runtime.h>
#include <stdint.h>
#include "fld_device.cuh"
using namespace fld;

__device__ unsigned long long g_wrong;

__device__ uint32_t mix(uint32_t x) {
    x ^= x >> 16; x *= 0x7feb352du; x ^= x >> 15; x *= 0x846ca68bu; x ^= x >> 16;
    return x;
}
__device__ bool same(float a, float b) { return __float_as_uint(a) == __float_as_uint(b); }
// 2^e (1 + m 2^-23)
__device__ float make(int e, uint32_t m) { return __uint_as_float(((uint32_t)(e + 127) << 23) | (m & 0x7fffffu)); }

// every mantissa times the exponents of quotient_range
__global__ void reciprocals(int exponent) {
    const uint32_t m = blockIdx.x * blockDim.x + threadIdx.x;
    if (m >= 1u << 23) return;
    const float b = make(exponent, m);
    if (!same(reciprocal_rn(b), __frcp_rn(b))) atomicAdd(&g_wrong, 1ull);
}

// D at random operands; edge: exponents at the ends of the ranges, one step inside,
// on and outside them, and mantissas of all zeros and ones among the random ones
__global__ void diffusion(uint32_t seed, int lim, int edge, uint32_t n) {
    const uint32_t t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= n) return;
    uint32_t r[8];
    for (int i = 0; i < 8; ++i) r[i] = mix(seed * 0x9e3779b9u + t * 8u + i);
    auto mantissa = [](uint32_t x, uint32_t how) { return how % 8 == 0 ? 0u : how % 8 == 1 ? 0x7fffffu : x; };
    auto exponent = [&](uint32_t x, int top) {
        const int end = (x & 1 ? 1 : -1) * top;
        return edge ? end - 1 + (int)((x >> 1) % 3) : (int)(x % (2u * top + 1u)) - top;
    };
    const float gmax = make(exponent(r[0], 50), mantissa(r[1], r[6]));
    const float sp = make(exponent(r[2], 20), mantissa(r[3], r[6] >> 3));
    // phi from a den of that range, or one close to gmax (R around 1 and up to 9)
    float den = make(exponent(r[4], 50), mantissa(r[5], r[6] >> 6));
    if (r[7] % 4 == 0) den = gmax * make(-(int)(r[7] >> 2) % 4, r[5]);
    const float phi = den / sp, floor_ = r[7] % 5 == 0 ? den : 1e-30f;
    const float a = D_of_f(D_point(gmax, sp), phi, floor_, lim, 2.0f);
    const float b = D_by_division(gmax, sp, phi, floor_, lim, 2.0f);
    if (!same(a, b)) atomicAdd(&g_wrong, 1ull);
}

extern "C" long long wrong_reciprocals(int exponent) {
    unsigned long long w = 0;
    if (cudaMemcpyToSymbol(g_wrong, &w, sizeof(w)) != cudaSuccess) return -1;
    reciprocals<<<(1 << 23) / 256, 256>>>(exponent);
    return cudaMemcpyFromSymbol(&w, g_wrong, sizeof(w)) == cudaSuccess ? (long long)w : -1;
}
extern "C" long long wrong_diffusion(unsigned seed, int lim, int edge, unsigned n) {
    unsigned long long w = 0;
    if (cudaMemcpyToSymbol(g_wrong, &w, sizeof(w)) != cudaSuccess) return -1;
    diffusion<<<(n + 255) / 256, 256>>>(seed, lim, edge, n);
    return cudaMemcpyFromSymbol(&w, g_wrong, sizeof(w)) == cudaSuccess ? (long long)w : -1;
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("quotients")
    src, so = d / "quotients.cu", d / "quotients.so"
    src.write_text(_CODE)
    r = subprocess.run([_build.nvcc(), *_build.ARCH, *_build.FLAGS, "-shared", "-o", str(so), str(src)],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    lib = ctypes.CDLL(str(so))
    for f in (lib.wrong_reciprocals, lib.wrong_diffusion):
        f.restype = ctypes.c_longlong
    return lib


@pytest.mark.parametrize("exponent", [-50, -20, -1, 0, 1, 20, 50])
def test_every_reciprocal(lib, exponent):
    assert lib.wrong_reciprocals(exponent) == 0


@pytest.mark.parametrize("limiter", ["lp", "kershaw", "larsen", "sum", "max", "cda"])
@pytest.mark.parametrize("edge", [0, 1])
def test_diffusion_coefficients(lib, limiter, edge):
    for seed in range(4):
        assert lib.wrong_diffusion(seed, fld.LIMITERS[limiter], edge, 1 << 26) == 0
