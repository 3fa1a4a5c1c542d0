"""Dense samples whose residuals take the one-launch FP64 path (products below
2^30 flops), at the edges of its 32 x 16 tiles and 16-deep slabs: n and L below,
at and above a multiple, one row, one column.  The refined samples match numpy's
FP64 solves of the same matrices to 1e-11 (backward errors reach 1e-14 after one
sweep of complex64 factors; the kernel's condition numbers stay below 1e3)."""
import numpy as np
import pytest

import oracle
import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rs():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1605_07951_gb300 import rsrr
    return rsrr


@pytest.mark.parametrize("n,L", [(2, 1), (16, 16), (17, 15), (31, 33), (32, 16), (33, 17), (64, 1), (129, 50)])
def test_refined_dense_samples(rs, n, L):
    p = W.helmholtz_sphere(n=n, N=5, L=L)
    s = rs.Solver(p, rs.default_opts(eta_tol=1e-14, max_refine=12))
    s.sample()
    S = s.samples()
    s.close()
    r = np.linalg.norm(p.points[:, None, :] - p.points[None, :, :], axis=2)
    np.fill_diagonal(r, 1.0)
    for j, z in enumerate(oracle.sample_points(p.region, p.N)):
        T = np.exp(1j * z * r) / (4.0 * np.pi * r)
        np.fill_diagonal(T, p.diag)
        X = np.linalg.solve(T, p.U)
        got = S[:, j * L:(j + 1) * L]
        assert np.linalg.norm(got - X) <= 1e-11 * np.linalg.norm(X)
