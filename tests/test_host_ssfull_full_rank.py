"""The host decomposition of SS-FULL where the Hankel matrix has full rank: its
pivoted QR then runs to the last column, behind which no column is left to update.
Built with the standard library's own bounds checks, so that an index past the end
of a vector ends the process; the eigenvalues are those of numpy's decomposition cut
at the same gap."""
import os
import shutil
import subprocess

import numpy as np
import pytest

from util import match_eigs

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = os.path.join(ROOT, "paper_1605_07951_gb300", "csrc")

HARNESS = r"""
#include <complex>
#include <cstdio>
#include <vector>
#include "ssfull_host.h"
int main(int argc, char **argv) {  // <moments> k KQ threads: eigenvalues to stdout
    using cplx = std::complex<double>;
    int k = 0, KQ = 0, threads = 0;
    sscanf(argv[2], "%d", &k);
    sscanf(argv[3], "%d", &KQ);
    sscanf(argv[4], "%d", &threads);
    std::vector<std::vector<cplx>> A(2 * KQ, std::vector<cplx>((size_t)k * k));
    FILE *f = fopen(argv[1], "rb");
    if (argc < 5 || !f) return 2;
    for (auto &a : A)
        if (fread(a.data(), sizeof(cplx), a.size(), f) != a.size()) return 2;
    fclose(f);
    std::vector<cplx> l, g;
    int nb = 0;
    double gm = 0.0;
    if (rsrr::ss_full_finish(A, k, KQ, cplx(0), 1.0, threads, l, g, nb, gm) != 0) return 3;
    for (int j = 0; j < nb; ++j) printf("%.17g %.17g\n", l[j].real(), l[j].imag());
    return 0;
}
"""


@pytest.fixture(scope="module")
def exe(tmp_path_factory):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no g++")
    d = tmp_path_factory.mktemp("ssfull_full_rank")
    h = d / "harness.cpp"
    h.write_text(HARNESS)
    out = d / "ssf"
    subprocess.run([gxx, "-O1", "-D_GLIBCXX_ASSERTIONS", "-std=c++17", "-fcx-fortran-rules", "-I", SRC, str(h),
                    os.path.join(SRC, "ssfull_host.cpp"), "-o", str(out), "-pthread"],
                   check=True, capture_output=True, text=True)
    return str(out)


@pytest.mark.parametrize("k,KQ", [(1, 1), (6, 1), (5, 2), (96, 1), (51, 2)])
def test_full_rank_moments(exe, tmp_path, k, KQ):
    ne = KQ * k
    rng = np.random.default_rng(10 * k + KQ)
    mom = rng.standard_normal((2 * KQ, k, k)) + 1j * rng.standard_normal((2 * KQ, k, k))
    hank = lambda o: np.block([[mom[i + j + o] for j in range(KQ)] for i in range(KQ)])
    H, Hs = hank(0), hank(1)
    if KQ == 1:  # prescribed singular values in (1, 2] and (0.01, 0.02]: one gap
        nb = max(1, 2 * ne // 3)
        U, _, Vh = np.linalg.svd(H)
        sv = np.concatenate([np.linspace(2, 1, nb, endpoint=False), np.linspace(0.02, 0.01, ne - nb, endpoint=False)])
        mom[0] = H = (U * sv) @ Vh
    U, sv, Vh = np.linalg.svd(H)
    assert sv[-1] > 1e-6 * sv[0]  # full rank, far above the rounding level where the decomposition stops
    nb = 1 if ne == 1 else 1 + int(np.argmax(sv[:-1] / sv[1:]))
    ref = np.linalg.eigvals(U[:, :nb].conj().T @ Hs @ Vh[:nb].conj().T / sv[:nb])
    path = tmp_path / "mom"
    np.ascontiguousarray(mom.transpose(0, 2, 1)).tofile(path)
    out = []
    for threads in (1, 4):
        r = subprocess.run([exe, str(path), str(k), str(KQ), str(threads)], capture_output=True, text=True)
        assert r.returncode == 0, (r.returncode, r.stderr)
        out.append(r.stdout)
    assert out[0] == out[1]
    lam = np.array([complex(*map(float, l.split())) for l in out[0].splitlines()])
    assert len(lam) == nb
    assert match_eigs(ref, lam) <= 1e-9
