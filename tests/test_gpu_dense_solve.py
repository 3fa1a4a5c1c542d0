"""Dense solves and the inverses of SS-FULL's nodes.

Solves: orders around the block size, point and probe counts that choose 4, 8 or
16 right-hand sides per chunk, ragged last chunks, and a matrix whose columns
all interchange rows.  The unrefined solutions' normwise backward errors, computed
here in numpy, stay below 8 n 2^-24 (2^-53 for FP64), Gaussian elimination's
bound with room for its growth factor.

SS-FULL: on a symmetric real problem with a contour symmetric about the real axis
one node of each conjugate pair is inverted; the eigenvalues agree with the
oracle's to 1e-9 for an even and an odd number of nodes, as they do for a centre
off the axis, where every node is inverted."""
import numpy as np
import pytest

import oracle
import workloads as W
from util import match_eigs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rs():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1605_07951_gb300 import rsrr
    return rsrr


@pytest.mark.parametrize("precision", [0, 1], ids=["fp64", "mixed"])
@pytest.mark.parametrize("n,N,L", [(5, 3, 2), (16, 3, 9), (33, 40, 33), (70, 20, 33), (129, 3, 18), (150, 130, 17)])
def test_unrefined_backward_error(rs, n, N, L, precision):
    q = W.dense_hidden_quadratic(n=n, N=N, L=L)
    perm = np.random.default_rng(n).permutation(n)  # pivots far from the diagonal
    q.As = [np.asfortranarray(A[perm]) for A in q.As]
    s = rs.Solver(q, rs.default_opts(precision=precision, max_refine=0))
    s.sample()
    S = s.samples()
    s.close()
    tol = 8.0 * n * (2.0 ** -53 if precision == 0 else 2.0 ** -24)
    z = oracle.sample_points(q.region, N)
    for j in (0, N // 2, N - 1):
        T = q.As[0] + z[j] * q.As[1] + z[j] ** 2 * q.As[2]
        X = S[:, j * L:(j + 1) * L]
        r = np.abs(q.U - T @ X).max(axis=0)
        eta = r / (np.abs(T).sum(axis=1).max() * np.abs(X).max(axis=0) + np.abs(q.U).max(axis=0))
        assert eta.max() <= tol, (j, eta.max(), tol)


@pytest.mark.parametrize("center,NQ", [(100.0, 128), (100.0, 129), (100.0 + 1.0j, 128)])
def test_eigenvalues_with_and_without_conjugate_nodes(rs, center, NQ):
    p = W.rational_grid(g=20, N=48, L=8, center=center)
    ref = oracle.rsrr(p, NQ=NQ, KQ=2)["lam"]
    s = rs.Solver(p, rs.default_opts(NQ=NQ, KQ=2, precision=rs.RSRR_PREC_FP64))
    s.sample()
    s.project()
    lam = s.solve()["lam"]
    s.close()
    assert len(lam) == len(ref) > 0
    assert match_eigs(ref, lam) <= 1e-9
