"""The refined square root, reciprocal and quotient of the exact arithmetic
(update.cuh) against CUDA's correctly rounded functions, bit for bit: root and
reciprocal for every fp32 value of the range in which the passes use them
(2^-100 to 2^100 under the root, 2^-60 to 2^60 for the reciprocal), the quotient
on pairs where a rounding can go wrong (the passes scale the dividend by 2^26 and
use quotients from 2^-40 to 2^120).  The kernels are compiled here, from the
header that the passes are compiled from."""

import subprocess

import pytest

from paper_1601_04033_gb300 import build

pytestmark = pytest.mark.gpu

SRC = r"""
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <cuda_runtime.h>
#include "kernels.cuh"
#include "update.cuh"
using namespace fasgd;
struct Result {
    unsigned long long wrong;
    float a, v, got, want;
};
__device__ void check(Result* r, float a, float v, float got, float want) {
    if (__float_as_uint(got) != __float_as_uint(want) && atomicAdd(&r->wrong, 1ull) == 0) {
        r->a = a; r->v = v; r->got = got; r->want = want;
    }
}
__device__ void quotient(Result* r, float a0, float a1, float v0, float v1) {
    const Pair v = pair(v0, v1);
    float x, y;
    unpack(minus_quotient2(pair(a0, a1), v, minus_reciprocal2(v)), x, y);
    check(r, a0, v0, -x, __fdiv_rn(a0, v0));
    check(r, a1, v1, -y, __fdiv_rn(a1, v1));
}
__device__ uint64_t mix(uint64_t x) {   // splitmix64
    x += 0x9E3779B97F4A7C15ull;
    x = (x ^ (x >> 30)) * 0xBF58476D1CE4E5B9ull;
    x = (x ^ (x >> 27)) * 0x94D049BB133111EBull;
    return x ^ (x >> 31);
}
// Bits of 2^-60 and 2^60, and a float of that range from 32 random bits and an exponent.
constexpr uint32_t kLo = 67u << 23, kHi = 187u << 23;
__device__ float in_range(uint32_t bits, uint32_t exponent) {
    return __uint_as_float((bits & 0x7fffffu) | ((67u + exponent % 120u) << 23));
}
__device__ uint32_t random_exponent(uint64_t h) { return (uint32_t)(h >> 40); }

// kind 0: root, 1: reciprocal, of the values from bits `from` on; 2: quotient of
// random pairs; 3: of a near v times a midpoint; 4: of all mantissas of a by the
// 1024 mantissas of v at both ends.
__global__ void sweep(int kind, uint64_t from, uint64_t n, Result* r) {
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
        float x, y;
        if (kind < 2) {   // the value and its neighbour at the other end of the range
            const float a = __uint_as_float((uint32_t)(from + i)), b = __uint_as_float((uint32_t)(from + n - 1 - i));
            if (kind == 0) {
                unpack(root2(pair(a, b), pair(-a, -b)), x, y);
                check(r, a, 0.f, x, __fsqrt_rn(a));
                check(r, b, 0.f, y, __fsqrt_rn(b));
            } else {
                unpack(minus_reciprocal2(pair(a, b)), x, y);
                check(r, a, 1.f, -x, __fdiv_rn(1.f, a));
                check(r, b, 1.f, -y, __fdiv_rn(1.f, b));
            }
            continue;
        }
        const uint64_t h = mix(from + 2 * i), g = mix(from + 2 * i + 1);
        const uint32_t sign = (uint32_t)(h >> 63) << 31;
        if (kind == 2) {
            quotient(r, __uint_as_float(__float_as_uint(in_range((uint32_t)h, random_exponent(h))) | sign),
                     in_range((uint32_t)g, random_exponent(g)), in_range((uint32_t)(h >> 23), random_exponent(g) >> 9),
                     in_range((uint32_t)(g >> 23), random_exponent(h) >> 9));
        } else if (kind == 5) {   // all exponents: of v, and of a for quotients from 2^-39 to 2^118
            const uint32_t ev = 67u + random_exponent(h) % 120u, eq = 88u + random_exponent(g) % 158u;
            const int ea = (int)eq + (int)ev - 127;
            if (ea < 1 || ea > 253) continue;
            const float a = __uint_as_float(((uint32_t)g & 0x7fffffu) | ((uint32_t)ea << 23) | sign);
            const float v = __uint_as_float(((uint32_t)h & 0x7fffffu) | (ev << 23));
            quotient(r, a, a, v, v);
        } else if (kind == 3) {
            // v in [1, 2), q in [1, 2) with a 25th bit set: a is the float next to
            // q v, so that a / v is as near to a midpoint as it gets; times powers of two.
            const float v = __uint_as_float(((uint32_t)h & 0x7fffffu) | (127u << 23));
            const double q = 1.0 + ((double)((uint32_t)g & 0x7fffffu) + 0.5) * 0x1p-23;
            const float a = __double2float_rn(q * (double)v), b = __uint_as_float(__float_as_uint(a) + ((g >> 32) & 1 ? 1 : -1));
            const float sa = __uint_as_float((127u - 58u + (uint32_t)(g >> 40) % 116u) << 23);
            const float sv = __uint_as_float((127u - 59u + (uint32_t)(h >> 40) % 118u) << 23);
            quotient(r, a * sa, b * sa, v * sv, v * sv);
        } else {
            const uint32_t k = (uint32_t)(i >> 23), m = k < 512 ? k : 0x800000u - 1u - (k - 512u);
            const float v = __uint_as_float(m | (127u << 23));
            const float a = __uint_as_float(((uint32_t)i & 0x7fffffu) | (127u << 23));
            quotient(r, a, a * 0x1p-59f, v, v * 0x1p59f);
        }
    }
}
__global__ void edges(Result* r) {   // zeros and both ends of the range, all pairs
    const uint32_t e[] = {0u, 0x80000000u, kLo, kLo + 1, kHi, kHi - 1, kLo | 0x80000000u, kHi | 0x80000000u, 127u << 23};
    for (uint32_t a : e)
        for (uint32_t v : e)
            if (v >= kLo && v <= kHi) quotient(r, __uint_as_float(a), __uint_as_float(a), __uint_as_float(v), __uint_as_float(v));
}
int main(int argc, char** argv) {
    const int kind = std::atoi(argv[1]);
    const uint64_t from = std::strtoull(argv[2], nullptr, 0), n = std::strtoull(argv[3], nullptr, 0);
    (void)argc;
    Result *r, h;
    if (cudaMalloc(&r, sizeof *r) != cudaSuccess || cudaMemset(r, 0, sizeof *r) != cudaSuccess) return std::printf("no memory\n"), 2;
    if (kind < 0)
        edges<<<1, 1>>>(r);
    else
        sweep<<<152 * 8, 256>>>(kind, from, n, r);
    if (cudaMemcpy(&h, r, sizeof h, cudaMemcpyDeviceToHost) != cudaSuccess) return std::printf("%s\n", cudaGetErrorString(cudaGetLastError())), 2;
    std::printf("%llu wrong; first: a = %a, v = %a, got %a, want %a\n", h.wrong, h.a, h.v, h.got, h.want);
    return h.wrong != 0;
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    d = tmp_path_factory.mktemp("sweep")
    (d / "sweep.cu").write_text(SRC)
    r = subprocess.run([build.nvcc(), *build.ARCH, "-std=c++17", "-O3", f"-I{build.INCLUDE}", f"-I{build.CSRC}",
                        str(d / "sweep.cu"), "-o", str(d / "sweep")], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return str(d / "sweep")


BITS = 1 << 23
SWEEPS = {"root": (0, 27 * BITS, 200 * BITS + 1), "reciprocal": (1, 67 * BITS, 120 * BITS + 1),
          "quotient random": (2, 12345, 1 << 34), "quotient near midpoints": (3, 999, 1 << 32),
          "quotient mantissas at the ends": (4, 0, 1024 * BITS), "quotient all exponents": (5, 777, 1 << 32), "quotient edges": (-1, 0, 0)}


@pytest.mark.parametrize("name", SWEEPS)
def test_correctly_rounded(program, name):
    r = subprocess.run([program, *map(str, SWEEPS[name])], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout + r.stderr
