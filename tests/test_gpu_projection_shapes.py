"""The projection over ranks and orders around its tiles: 32-row blocks of the
pivoted Cholesky, odd and even orders and few or many pairs of the Jacobi rounds,
results of at most and of more than 48 columns of the FP64 products."""
import numpy as np
import pytest

import oracle
import workloads as W

pytestmark = pytest.mark.gpu


# order g^2, moment columns 2 * 2 * L before the rank is found
@pytest.mark.parametrize("g,L", [(2, 1), (3, 2), (5, 4), (6, 9), (8, 16), (9, 13), (13, 24), (16, 33)])
def test_basis_and_projected_coefficients(g, L):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1605_07951_gb300 import rsrr as rs
    p = W.rational_grid(g=g, N=16, L=L)
    s = rs.Solver(p, rs.default_opts(NQ=32, KQ=2, gemm=1))
    s.sample()
    s.check()
    s.project()
    Q, P = s.Q(), s.projected()
    s.close()
    k = Q.shape[1]
    assert 1 <= k <= g * g
    # two Gram passes leave an orthogonality error of a few eps * k
    assert np.abs(Q.conj().T @ Q - np.eye(k)).max() <= 1e-12
    for i, (Pg, Pr) in enumerate(zip(P, oracle.project(p, Q))):
        a1 = np.abs(oracle.coeff_matrix(p, i)).sum(axis=0).max()
        assert np.abs(Pg - Pr).max() <= 1e-13 * max(a1, 1e-300), i
