"""Sliced products with more tiles than SMs, so that a CTA's ring of stages and its
tensor-memory folds run on from tile to tile: depths of one stage, of exactly one
fold, of one stage more and of several folds, results added to C with a sign, and
Hermitian results whose lower tiles are left out.  Integer inputs, for which every sum
is exact in FP64, so the product must be exact bit for bit."""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def product(A, B, C0, conjA, hermitian, alpha, beta):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1605_07951_gb300 import rsrr
    M, K = (A.shape[1], A.shape[0]) if conjA else A.shape
    d = [torch.from_numpy(np.ascontiguousarray(X.T)).to("cuda") for X in (A, B, C0)]
    if hermitian:
        d[1] = d[0]
    p = [ctypes.c_void_p(t.data_ptr()) for t in d]
    st = rsrr.rsrr_zgemm(M, B.shape[1], K, int(conjA), p[0], A.shape[0], p[1], B.shape[0], p[2], M, alpha, beta, 2,
                         int(hermitian), 0, None)
    assert st == rsrr.RSRR_OK, rsrr.rsrr_last_error(None).decode()
    return d[2].cpu().numpy().T


def integers(rng, *s):
    return (rng.integers(-1000, 1001, s) + 1j * rng.integers(-1000, 1001, s)).astype(np.complex128)


@pytest.mark.parametrize("M,N,K", [(20000, 33, 8), (20010, 40, 96), (9999, 70, 97), (5000, 129, 300)])
def test_many_tiles_per_cta(M, N, K):
    rng = np.random.default_rng(M + K)
    A, B, C0 = integers(rng, M, K), integers(rng, K, N), 2.0 * integers(rng, M, N)
    assert np.array_equal(product(A, B, C0, False, False, -1.0, 0.5), 0.5 * C0 - A @ B)


@pytest.mark.parametrize("N,K", [(100, 3000), (700, 96), (833, 97), (1500, 200)])
def test_hermitian_tiles(N, K):
    rng = np.random.default_rng(N + K)
    A = integers(rng, K, N)
    assert np.array_equal(product(A, A, np.zeros((N, N), complex), True, True, 1.0, 0.0), A.conj().T @ A)
