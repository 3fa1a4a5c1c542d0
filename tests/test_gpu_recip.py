"""The band LU's fast reciprocals (recip.cuh) against CUDA's own division, bit by
bit, in a program compiled here with the library's flags:

  * real: every float of 2^-41 .. 2^42, both signs (the complex form divides by
    sums up to 2^41);
  * complex against crecip(): the larger component at exponents across the range
    and both its ends, the smaller one at every ratio 2^0 .. 2^-50, either order,
    all signs, with random mantissas and with all pairs of mantissas next to powers
    of two, to their middle and to the places where rounded reciprocals turn; and
    with the smaller component zero of either sign;
  * ok, which says whether the fast form applies: true inside the stated range up to
    its ends, false just outside, for zeros, infinities, NaN and subnormals."""
import os
import subprocess

import pytest

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include <cstdio>
#include "recip.cuh"
using namespace rsrr;

__device__ unsigned long long g_bad[4], g_all[4];
__device__ unsigned hash32(unsigned x) {
    x ^= x >> 16; x *= 0x7feb352du; x ^= x >> 15; x *= 0x846ca68bu; x ^= x >> 16;
    return x;
}
__device__ void add(int k, unsigned long long bad, unsigned long long all) {
    atomicAdd(&g_bad[k], bad);
    atomicAdd(&g_all[k], all);
}
// exponents 127 - 41 .. 127 + 41 (up to 2^42), every mantissa, both signs
__global__ void real_all() {
    const unsigned lo = (127u - 41u) << 23, hi = (127u + 42u) << 23;
    unsigned long long bad = 0, all = 0;
    for (unsigned u = lo + blockIdx.x * blockDim.x + threadIdx.x; u < hi; u += gridDim.x * blockDim.x)
        for (unsigned s = 0; s < 2; ++s) {
            const float b = __uint_as_float(u | (s << 31));
            bad += __float_as_uint(recip_rn(b)) != __float_as_uint(crecip(b));
            ++all;
        }
    add(0, bad, all);
}
__device__ bool same(float2 b) {
    bool ok;
    const float2 y = recip_fast(b, ok), c = crecip(b);
    return ok && __float_as_uint(y.x) == __float_as_uint(c.x) && __float_as_uint(y.y) == __float_as_uint(c.y);
}
__constant__ int c_exp[] = {-40, -39, -20, -1, 0, 1, 17, 38, 39};
__device__ unsigned special(int i) {  // 64 mantissas
    const unsigned m[8] = {0u, 0x7fffffu, 0x400000u, 0x3fffffu, 0x2aaaaau, 0x555555u, 0x3504f3u, 0x5a8279u};
    return (m[i & 7] + (unsigned)(i >> 3)) & 0x7fffffu;
}
// one exponent and ratio a block row; random mantissas, then the special ones
__global__ void complex_pairs(unsigned draws) {
    const int e = c_exp[blockIdx.y % 9], s = blockIdx.y / 9;  // s = 0 .. 50
    const unsigned step = gridDim.x * blockDim.x, first = blockIdx.x * blockDim.x + threadIdx.x;
    unsigned long long bad = 0, all = 0;
    for (unsigned i = first; i < draws + 4096u; i += step) {
        const unsigned h = hash32(i * 977u + blockIdx.y * 0x9e3779b9u), g = hash32(h + 0x85ebca6bu);
        unsigned mb = h >> 9, ms = g >> 9;
        if (i >= draws) {
            mb = special((i - draws) & 63);
            ms = special((i - draws) >> 6);
        }
        // (the ratio of the components stays within 1 .. 2^50: their mantissas in order at both ends)
        if ((s == 0 && ms > mb) || (s == 50 && ms < mb)) { const unsigned t = mb; mb = ms; ms = t; }
        const float big = __uint_as_float(((unsigned)(127 + e) << 23) | mb | (h << 31));
        const float small = __uint_as_float(((unsigned)(127 + e - s) << 23) | ms | (g << 31));
        bad += !same((g & 2) ? make_float2(big, small) : make_float2(small, big));
        ++all;
    }
    add(1, bad, all);
}
__global__ void complex_zero() {
    unsigned long long bad = 0, all = 0;
    for (unsigned i = blockIdx.x * blockDim.x + threadIdx.x; i < (1u << 23); i += gridDim.x * blockDim.x)
        for (int q = 0; q < 9; ++q)
            for (unsigned v = 0; v < 8; ++v) {
                const float big = __uint_as_float(((unsigned)(127 + c_exp[q]) << 23) | i | (v << 31));
                const float zero = __uint_as_float((v >> 1) << 31);
                bad += !same((v & 4) ? make_float2(big, zero) : make_float2(zero, big));
                ++all;
            }
    add(2, bad, all);
}
__global__ void ranges() {
    const float lo = __uint_as_float((127u - 40u) << 23), hi = __uint_as_float((127u + 40u) << 23);
    const float in[] = {lo, hi, 1.f, 3.f}, inf = __uint_as_float(0x7f800000u), nan = __uint_as_float(0x7fc00000u);
    const float out[] = {__uint_as_float(__float_as_uint(lo) - 1u), __uint_as_float(__float_as_uint(hi) + 1u), 0.f, inf, nan,
                         __uint_as_float(1u), 1e-40f};
    unsigned long long bad = 0, all = 0;
    bool ok;
    for (float sg = 1.f; sg >= -1.f; sg -= 2.f) {
        for (float v : in) {
            recip_fast(sg * v, ok); bad += !ok;
            recip_fast(make_float2(sg * v, 0.f), ok); bad += !ok;
            recip_fast(make_float2(v * 0x1p-50f, sg * v), ok); bad += !ok;
            recip_fast(make_float2(sg * v, __uint_as_float(__float_as_uint(v * 0x1p-50f) - 1u)), ok); bad += ok;
            recip_fast(make_float2(v, sg * nan), ok); bad += ok;
            all += 5;
        }
        for (float v : out) {
            recip_fast(sg * v, ok); bad += ok;
            recip_fast(make_float2(sg * v, 0.f), ok); bad += ok;
            recip_fast(make_float2(0.f, sg * v), ok); bad += ok;
            all += 3;
        }
        recip_fast(make_float2(1.f, sg * inf), ok); bad += ok;
        recip_fast(make_float2(sg * nan, 1.f), ok); bad += ok;
        all += 2;
    }
    add(3, bad, all);
}
int main() {
    real_all<<<1216, 256>>>();
    complex_pairs<<<dim3(64, 9 * 51), 256>>>(1u << 22);
    complex_zero<<<1216, 256>>>();
    ranges<<<1, 1>>>();
    unsigned long long bad[4], all[4];
    cudaError_t e = cudaMemcpyFromSymbol(bad, g_bad, sizeof bad);
    if (e == cudaSuccess) e = cudaMemcpyFromSymbol(all, g_all, sizeof all);
    if (e != cudaSuccess) { fprintf(stderr, "%s\n", cudaGetErrorString(e)); return 1; }
    for (int k = 0; k < 4; ++k) printf("%llu %llu\n", bad[k], all[k]);
    return 0;
}
"""


def test_same_bits_as_division(tmp_path):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1605_07951_gb300 import build
    src = tmp_path / "recip_test.cu"
    src.write_text(SOURCE)
    exe = str(tmp_path / "recip_test")
    subprocess.run([build.nvcc()] + build.ARCH + build.FLAGS + [str(src), "-o", exe], check=True, capture_output=True,
                   text=True)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr
    bad, count = zip(*[tuple(map(int, l.split())) for l in r.stdout.splitlines()])
    assert count[0] == 2 * 83 * 2 ** 23
    assert count[1] == 9 * 51 * (2 ** 22 + 4096)
    assert count[2] == 8 * 9 * 2 ** 23
    assert bad == (0, 0, 0, 0)
