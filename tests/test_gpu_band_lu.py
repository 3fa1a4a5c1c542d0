"""Band LU at the edges of its kernel instances: lower half-bandwidths on both
sides of each instance's limit (32, 64, 128, 224), panels that take every warp
(kl > 448), bands without a lower or an upper part, n off the block size, and
matrices whose weak diagonal makes most columns interchange rows.

The unrefined solutions' normwise backward errors, computed here in numpy, stay
below 8 (2 kl + ku + 1) 2^-24 (2^-53 for FP64): the usual bound of Gaussian
elimination with partial pivoting grows with the rows an element meets, and a
factor 8 leaves room for the growth factor of random matrices.  One CTA and a
cluster of CTAs per point give the same bits."""
import numpy as np
import pytest

import oracle
import workloads as W

pytestmark = pytest.mark.gpu

SHAPES = [(5, 1, 1), (33, 0, 3), (45, 3, 0), (97, 31, 4), (130, 32, 32), (131, 33, 64), (200, 64, 1), (260, 65, 40),
          (300, 128, 20), (301, 129, 128), (420, 224, 9), (421, 225, 30), (1000, 449, 12), (1025, 480, 3)]


@pytest.fixture(scope="module")
def rs():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1605_07951_gb300 import rsrr
    return rsrr


@pytest.mark.parametrize("n,kl,ku", SHAPES, ids=["n%d_kl%d_ku%d" % s for s in SHAPES])
@pytest.mark.parametrize("precision", [0, 1], ids=["fp64", "mixed"])
def test_unrefined_backward_error(rs, n, kl, ku, precision):
    p = W.random_banded(n=n, kl=kl, ku=ku, N=3, L=2, seed=100 + n)
    rows = np.repeat(np.arange(n), np.diff(p.row_ptr))
    p.values[0] = np.where(rows == p.col_idx, 0.05 * p.values[0], p.values[0])
    S = []
    for flags in (0, rs.RSRR_FLAG_ONE_CTA_LU):
        s = rs.Solver(p, rs.default_opts(precision=precision, max_refine=0, flags=flags))
        s.sample()
        S.append(s.samples().copy())
        s.close()
    assert np.array_equal(S[0], S[1])
    tol = 8.0 * (2 * kl + ku + 1) * (2.0 ** -53 if precision == 0 else 2.0 ** -24)
    for j, z in enumerate(oracle.sample_points(p.region, p.N)):
        T = np.zeros((n, n), dtype=np.complex128)
        T[rows, p.col_idx] = p.values[0] + z * p.values[1] + z * z * p.values[2]
        X = S[0][:, j * p.L:(j + 1) * p.L]
        r = np.abs(p.U - T @ X).max(axis=0)
        eta = r / (np.abs(T).sum(axis=1).max() * np.abs(X).max(axis=0) + np.abs(p.U).max(axis=0))
        assert eta.max() <= tol, (j, eta.max(), tol)
