"""Assembly of the dense kernel matrix by pairs of 32 x 32 tiles and its row-sum
norm: orders around the tile size, one point and enough points that a block takes
several.  FP64 samples solve the oracle's T(z) to a backward error of 1e-14, and the
reported backward error (which divides by the norm) is the oracle's."""
import numpy as np
import pytest

import oracle
import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,N", [(12, 1), (31, 5), (32, 2), (33, 3), (64, 1), (65, 2), (97, 1300), (400, 70)])
def test_samples_and_backward_errors(n, N):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1605_07951_gb300 import rsrr as rs
    L = 2
    p = W.helmholtz_sphere(n=n, N=N, L=L)
    s = rs.Solver(p, rs.default_opts(precision=rs.RSRR_PREC_FP64))
    s.sample()
    assert s.check_status() == rs.RSRR_OK
    S, eta = s.samples(), s.eta()
    s.close()
    zo = oracle.sample_points(p.region, p.N)
    for j in sorted({0, N // 2, N - 1}):
        e = oracle.backward_error_inf_dense(p, zo[j], S[:, j * L:(j + 1) * L])
        assert e.max() <= 1e-14
        assert np.allclose(eta[j * L:(j + 1) * L], e, rtol=1e-3, atol=1e-14)
