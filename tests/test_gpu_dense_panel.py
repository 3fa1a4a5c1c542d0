"""Panels of the dense LU: rows on either side of 256, 512, 1024, 2048 and 4096,
where the rows held by a thread and the columns taken at a time change, ragged last
panels, interchanges in every column.  The unrefined solutions' normwise backward
errors, computed here in numpy, stay below 8 n 2^-24 (2^-53 for FP64), Gaussian
elimination's bound with room for its growth factor."""
import numpy as np
import pytest

import oracle
import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [0, 1], ids=["fp64", "mixed"])
@pytest.mark.parametrize("n,N", [(1, 2), (31, 3), (250, 3), (261, 160), (515, 3), (530, 2), (1045, 2), (2061, 2), (4103, 1)])
def test_unrefined_backward_error(n, N, precision):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1605_07951_gb300 import rsrr as rs
    L = 3
    q = W.dense_hidden_quadratic(n=8, N=N, L=L)
    rng = np.random.default_rng(n)
    d = [rng.standard_normal((n, n)) for _ in range(2)]
    q.As = [np.asfortranarray(m.astype(complex)) for m in (d[0], d[1], np.eye(n))]
    q.n = n
    q.U = np.asfortranarray(rng.standard_normal((n, L)) + 1j * rng.standard_normal((n, L)))
    s = rs.Solver(q, rs.default_opts(precision=precision, max_refine=0))
    s.sample()
    S = s.samples()
    s.close()
    tol = 8.0 * n * (2.0 ** -53 if precision == 0 else 2.0 ** -24)
    z = oracle.sample_points(q.region, N)
    for j in sorted({0, N // 2, N - 1}):
        T = q.As[0] + z[j] * q.As[1] + z[j] ** 2 * q.As[2]
        X = S[:, j * L:(j + 1) * L]
        r = np.abs(q.U - T @ X).max(axis=0)
        eta = r / (np.abs(T).sum(axis=1).max() * np.abs(X).max(axis=0) + np.abs(q.U).max(axis=0))
        assert eta.max() <= tol, (j, eta.max(), tol)
