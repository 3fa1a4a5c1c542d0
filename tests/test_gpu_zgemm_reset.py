"""rsrr_zgemm works before and after a cudaDeviceReset: the same product has the same
bits, two resets in a row, and what the call keeps on the device (its pool is not
among the resources that a reset destroys) is given back as before it, when a handle
is created.  In a process of its own, whose only use of CUDA is through the runtime."""
import os
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

pytestmark = pytest.mark.gpu

CODE = r"""
import ctypes as C
import numpy as np
import workloads as W
from paper_1605_07951_gb300 import rsrr

rt = None  # the runtime that the library is linked with
for line in open("/proc/self/maps"):
    path = line.split()[-1]
    if "libcudart.so" in path:
        rt = C.CDLL(path)
        break
def ok(e):
    assert e == 0, e
def free():
    a, b = C.c_size_t(), C.c_size_t()
    ok(rt.cudaMemGetInfo(C.byref(a), C.byref(b)))
    return a.value
M, K = 200, 30000
rng = np.random.default_rng(3)
A = rng.standard_normal((M, K)) + 1j * rng.standard_normal((M, K))
held = []
def product():
    dA, dC = C.c_void_p(), C.c_void_p()
    ok(rt.cudaMalloc(C.byref(dA), C.c_size_t(A.nbytes)))
    ok(rt.cudaMalloc(C.byref(dC), C.c_size_t(16 * M * M)))
    ok(rt.cudaMemcpy(dA, A.ctypes.data_as(C.c_void_p), C.c_size_t(A.nbytes), 1))
    for _ in range(2):
        st = rsrr.rsrr_zgemm(M, M, K, 1, dA, K, dA, K, dC, M, 1.0, 0.0, rsrr.RSRR_GEMM_AUTO, 1, 0, None)
        assert st == rsrr.RSRR_OK, rsrr.rsrr_last_error(None)
    G = np.empty((M, M), dtype=np.complex128)
    ok(rt.cudaMemcpy(G.ctypes.data_as(C.c_void_p), dC, C.c_size_t(G.nbytes), 2))
    held[:] = [dA, dC]
    return G
ok(rt.cudaFree(None))
start = free()
ref = product()
assert abs(ref[3, 3].real - (np.abs(A[3]) ** 2).sum()) < 1e-8 * K
for _ in range(2):
    ok(rt.cudaDeviceReset())
    ok(rt.cudaFree(None))
    assert np.array_equal(product(), ref)
    assert start - free() > 300 << 20  # the matrices of the product, and what the call keeps
    ok(rt.cudaFree(held.pop()))
    ok(rt.cudaFree(held.pop()))
    rsrr.Solver(W.random_banded(n=20, kl=1, ku=1, N=1, L=1)).close()
    ok(rt.cudaDeviceSynchronize())
    print(start - free())
    assert start - free() < 128 << 20, (free(), start)
print("ok")
"""


def test_product_after_reset():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    r = subprocess.run([sys.executable, "-c", CODE], cwd=ROOT, capture_output=True, text=True, timeout=300,
                       env=dict(os.environ, PYTHONPATH=ROOT))
    assert r.returncode == 0 and r.stdout.strip().endswith("ok"), (r.returncode, r.stdout, r.stderr[-2000:])
