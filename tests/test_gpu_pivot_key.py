"""Keys of the band LU's pivot search, in a program compiled here with the library's
flags: they order |re| + |im| as the numbers do, infinities last, and count a NaN as
zero, as the comment at them says, although a compiler that takes a sum of moduli for
non-negative may drop a comparison that is there for NaN.  No key is 0, which stands
for rows that are no candidates."""
import subprocess

import pytest

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include <cstdio>
#define RSRR_LU_ONLY 0
#include "band_lu.cu"
using namespace rsrr;
__device__ int g_bad[4];
template <typename C, typename R> __device__ void check(const R *v, int n, int slot, C (*make)(R, R)) {
    // v: ascending moduli, the last three NaN (quiet, as arithmetic leaves them, of either sign)
    int bad = 0;
    for (int i = 0; i < n; ++i)
        for (int j = 0; j < n; ++j) {
            const auto a = pivot_key(cabs1(make(v[i], R(0)))), b = pivot_key(cabs1(make(R(0), -v[j])));
            const bool na = i >= n - 3, nb = j >= n - 3;
            if (a == 0 || b == 0) ++bad;
            if (na && a != pivot_key(R(0))) ++bad;
            if (!na && !nb && ((v[i] < v[j]) != (a < b) || (v[i] == v[j]) != (a == b))) ++bad;
            if (na && !nb && a > b) ++bad;
        }
    g_bad[slot] = bad;
}
__device__ float2 cf(float a, float b) { return make_float2(a, b); }
__device__ double2 cd(double a, double b) { return make_double2(a, b); }
__device__ float rf(float a, float b) { return a + b; }
__device__ double rd(double a, double b) { return a + b; }
__global__ void run(const float *f, const double *d, int n) {
    check<float2, float>(f, n, 0, cf);
    check<double2, double>(d, n, 1, cd);
    check<float, float>(f, n, 2, rf);
    check<double, double>(d, n, 3, rd);
}
int main() {
    const unsigned fb[] = {0u, 1u, 0x00800000u, 0x3f800000u, 0x3f800001u, 0x7f7fffffu, 0x7f800000u, 0x7fffffffu, 0xffc00000u, 0x7fc00001u};
    const unsigned long long db[] = {0ull, 1ull, 0x0010000000000000ull, 0x3ff0000000000000ull, 0x3ff0000000000001ull,
                                     0x7fefffffffffffffull, 0x7ff0000000000000ull, 0x7fffffffffffffffull, 0xfff8000000000000ull,
                                     0x7ff8000000000001ull};
    float *f = nullptr;
    double *d = nullptr;
    int bad[4];
    cudaError_t e = cudaMalloc(&f, sizeof fb);
    if (e == cudaSuccess) e = cudaMalloc(&d, sizeof db);
    if (e == cudaSuccess) e = cudaMemcpy(f, fb, sizeof fb, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemcpy(d, db, sizeof db, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) run<<<1, 1>>>(f, d, 10);
    if (e == cudaSuccess) e = cudaMemcpyFromSymbol(bad, g_bad, sizeof bad);
    if (e != cudaSuccess) { fprintf(stderr, "%s\n", cudaGetErrorString(e)); return 1; }
    printf("%d %d %d %d\n", bad[0], bad[1], bad[2], bad[3]);
    return 0;
}
"""


def test_keys(tmp_path):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1605_07951_gb300 import build
    src = tmp_path / "key_test.cu"
    src.write_text(SOURCE)
    exe = str(tmp_path / "key_test")
    subprocess.run([build.nvcc()] + build.ARCH + build.FLAGS + [str(src), "-o", exe], check=True, capture_output=True,
                   text=True)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stderr
    assert r.stdout.split() == ["0"] * 4
