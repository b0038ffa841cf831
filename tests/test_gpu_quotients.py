"""The short division sequence against exact remainders: for a, b in [1, 2) the
remainder a - b q of a quotient within one unit is a binary32 number, so one FMA
gives it exactly, and q is correctly rounded where |a - b q| <= b ulp(q) / 2.
Every numerator significand over 8,192 divisors spread over all; all 2^46 pairs
with GPFDP_ALL_QUOTIENTS=1 in the environment (36 s).  The machine's
reciprocal approximation has to have the same significand at every exponent of
the sequence's range, so that the scale of the operands changes no bit."""
import ctypes
import os
import subprocess

import pytest

pytestmark = pytest.mark.gpu

SRC = r"""
#include "interp.cuh"
// block: a divisor; threads: its 2^23 numerators, four quotients at a time
__global__ void quotients(uint32_t first, uint32_t step, unsigned long long* bad) {
    const uint32_t bm = (first + blockIdx.x * step) & 0x7FFFFFu;
    const float b = __uint_as_float(0x3F800000u | bm);
    uint32_t n = 0;
    for (uint32_t am = 4 * threadIdx.x; am < (1u << 23); am += 4 * blockDim.x) {
        float q[4], d[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) { q[k] = __uint_as_float(0x3F800000u | (am + k)); d[k] = b; }
        pdiv_vec<4>(q, d);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const float a = __uint_as_float(0x3F800000u | (am + k));
            const float per_half_unit = am + k >= bm ? 16777216.0f : 33554432.0f;
            n += !(fabsf(__fmaf_rn(-b, q[k], a)) * per_half_unit <= b);
        }
    }
    if (n) atomicAdd(bad, (unsigned long long)n);
}
__global__ void exponents(unsigned long long* bad) {
    const uint32_t bm = blockIdx.x * blockDim.x + threadIdx.x;
    float y, z;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(__uint_as_float(0x3F800000u | bm)));
    uint32_t n = 0;
    for (int x = -60; x <= 60; ++x) {
        const uint32_t b = (uint32_t)(127 + x) << 23 | bm, want = __float_as_uint(y) - ((uint32_t)x << 23);
        asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(z) : "f"(__uint_as_float(b)));
        n += __float_as_uint(z) != want;
        asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(z) : "f"(__uint_as_float(b | 0x80000000u)));
        n += __float_as_uint(z) != (want | 0x80000000u);
    }
    if (n) atomicAdd(bad, (unsigned long long)n);
}
extern "C" int run(uint32_t first, uint32_t step, uint32_t divisors, int check_exponents, unsigned long long* out) {
    unsigned long long* d;
    if (cudaMalloc(&d, 8) != cudaSuccess || cudaMemset(d, 0, 8) != cudaSuccess) return 1;
    if (check_exponents) exponents<<<(1u << 23) / 256, 256>>>(d);
    else quotients<<<divisors, 256>>>(first, step, d);
    const bool ok = cudaGetLastError() == cudaSuccess && cudaMemcpy(out, d, 8, cudaMemcpyDeviceToHost) == cudaSuccess;
    cudaFree(d);
    return ok ? 0 : 2;
}
"""


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    from paper_2205_03251_gb300 import _build
    d = tmp_path_factory.mktemp("quotients")
    (d / "quotients.cu").write_text(SRC)
    lib = d / "quotients.so"
    subprocess.check_call([_build._nvcc(), *_build.NVCC_FLAGS, "-I", _build.INCLUDE, "-I", _build.CSRC, "-o", str(lib),
                           str(d / "quotients.cu")])
    so = ctypes.CDLL(str(lib))

    def call(first, step, divisors, exponents=0):
        bad = ctypes.c_ulonglong(1)
        assert so.run(ctypes.c_uint32(first), ctypes.c_uint32(step), ctypes.c_uint32(divisors), exponents,
                      ctypes.byref(bad)) == 0
        return bad.value
    return call


def test_reciprocal_is_the_same_at_every_exponent(run):
    assert run(0, 1, 1, 1) == 0


def test_every_quotient_is_correctly_rounded(run):
    assert run(0, 2048, 4096) == 0
    assert run(1 + 777, 2048, 4096) == 0
    if os.environ.get("GPFDP_ALL_QUOTIENTS"):
        for first in range(0, 1 << 23, 8192):
            assert run(first, 1, 8192) == 0, first
