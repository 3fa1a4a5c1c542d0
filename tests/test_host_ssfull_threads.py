"""The host decomposition of SS-FULL with one and with several threads: columns of a
step go to threads by fours, so sizes around that and around the size at which a
second thread starts (8192 elements) give the same eigenvalues to the last bit, and
the eigenvalues are those the moments were made of."""
import ctypes as C
import os
import shutil
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = os.path.join(ROOT, "paper_1605_07951_gb300", "csrc")

HARNESS = r"""
#include <complex>
#include <vector>
#include "ssfull_host.h"
extern "C" int ssf(const double *mom, int k, int KQ, int threads, int cap, double *lam) {
    using cplx = std::complex<double>;
    std::vector<std::vector<cplx>> A(2 * KQ, std::vector<cplx>((size_t)k * k));
    for (int a = 0; a < 2 * KQ; ++a)
        for (size_t e = 0; e < (size_t)k * k; ++e)
            A[a][e] = cplx(mom[2 * ((size_t)a * k * k + e)], mom[2 * ((size_t)a * k * k + e) + 1]);
    std::vector<cplx> l, g;
    int nb = 0;
    double gm = 0.0;
    if (rsrr::ss_full_finish(A, k, KQ, cplx(0), 1.0, threads, l, g, nb, gm) != 0 || nb > cap) return -1;
    for (int j = 0; j < nb; ++j) { lam[2 * j] = l[j].real(); lam[2 * j + 1] = l[j].imag(); }
    return nb;
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no g++")
    d = tmp_path_factory.mktemp("ssfull_threads")
    h = d / "harness.cpp"
    h.write_text(HARNESS)
    so = d / "libssf.so"
    subprocess.run([gxx, "-O2", "-std=c++17", "-shared", "-fPIC", "-fcx-fortran-rules", "-I", SRC, str(h),
                    os.path.join(SRC, "ssfull_host.cpp"), "-o", str(so), "-pthread"],
                   check=True, capture_output=True, text=True)
    L = C.CDLL(str(so))
    L.ssf.argtypes = [C.c_void_p, C.c_int, C.c_int, C.c_int, C.c_int, C.c_void_p]
    return L


@pytest.mark.parametrize("k,ne", [(1, 1), (5, 3), (45, 7), (46, 8), (65, 33), (99, 12)])
def test_threads_give_the_same_bits(lib, k, ne):
    KQ = 2
    rng = np.random.default_rng(k)
    X = rng.standard_normal((k, ne)) + 1j * rng.standard_normal((k, ne))
    Y = rng.standard_normal((k, ne)) + 1j * rng.standard_normal((k, ne))
    s = np.linspace(-0.9, 0.9, ne) + 0.05j
    mom = np.stack([(X * s ** al) @ Y.conj().T for al in range(2 * KQ)])
    buf = np.ascontiguousarray(mom.transpose(0, 2, 1))  # column major per moment
    out = []
    for threads in (1, 2, 7):
        lam = np.zeros(2 * k, dtype=complex)
        nb = lib.ssf(buf.ctypes.data, k, KQ, threads, 2 * k, lam.ctypes.data)
        assert nb == ne
        out.append(lam[:nb])
    assert all(np.array_equal(out[0], o) for o in out[1:])
    # the lifted problem is as conditioned as X and Y: far inside 1e-9
    assert max(np.abs(out[0] - e).min() for e in s) <= 1e-9
