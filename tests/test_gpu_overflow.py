"""Matrices that are finite in double precision and overflow in complex64: a column of
T(z) is infinite in the mixed path's factor at one of two sampling points, the rest of
that factor becomes NaN, and no candidate of a pivot is a number any more.  Every LU
(a band by one CTA and by a cluster, in real arithmetic, dense panels in registers and
in global memory) ends with pivots inside the matrix: the other point's samples are as
accurate as without, the point itself is reported, and the FP64 path solves both."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rs():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1605_07951_gb300 import rsrr
    return rsrr


def both_paths(rs, p, T, real=False):
    """p at the points 0 (where nothing overflows) and 1/2; T(z) dense."""
    flags = rs.RSRR_FLAG_REAL if real else 0
    for precision in (rs.RSRR_PREC_MIXED, rs.RSRR_PREC_FP64):
        s = rs.Solver(p, rs.default_opts(precision=precision, flags=flags))
        s.sample()
        st, S, z = s.check_status(), s.samples().copy(), s.points()
        s.close()
        for j in range(2):
            if precision == rs.RSRR_PREC_MIXED and z[j] != 0:
                assert st in (rs.RSRR_ENOCONV, rs.RSRR_ESINGULAR)
                continue
            A, X = T(z[j]), S[:, j * p.L:(j + 1) * p.L]
            r = np.abs(p.U - A @ X).max(axis=0)
            eta = r / (np.abs(A).sum(axis=1).max() * np.abs(X).max(axis=0) + np.abs(p.U).max(axis=0))
            assert eta.max() <= 1e-10, (precision, j, eta.max())
        if precision == rs.RSRR_PREC_FP64:
            assert st == rs.RSRR_OK


@pytest.mark.parametrize("n,kl,ku,real", [(20, 2, 3, False), (70, 2, 3, False), (200, 40, 40, False), (700, 240, 240, False), (90, 5, 5, True)])
def test_band(rs, n, kl, ku, real):
    p = W.random_banded(n=n, kl=kl, ku=ku, m=2, N=2, L=3, seed=n)
    rows = np.repeat(np.arange(n), np.diff(p.row_ptr))
    p.values[1] = np.where(p.col_idx == n // 2, 1e39 * p.values[1], p.values[1])
    p.region = W.Region(0.25, 0.5, 0.4, kind="points", points=np.array([0.0, 0.5], dtype=complex))
    if real:
        p.U = np.asfortranarray(p.U.real.astype(np.complex128))

    def T(z):
        A = np.zeros((n, n), dtype=np.complex128)
        A[rows, p.col_idx] = p.values[0] + z * p.values[1]
        return A

    both_paths(rs, p, T, real)


class Terms:
    pass


@pytest.mark.parametrize("n", [40, 130, 900, 4200])
def test_dense(rs, n):
    rng = np.random.default_rng(n)
    p = Terms()
    p.n, p.N, p.L = n, 2, 3
    A0 = rng.standard_normal((n, n)) + 1j * rng.standard_normal((n, n))
    A0[np.arange(n), np.arange(n)] += 8.0 * np.sqrt(n)
    A1 = np.zeros((n, n), dtype=np.complex128)
    A1[:, n // 2] = 1e39 * (rng.standard_normal(n) + 1j * rng.standard_normal(n))
    p.As, p.fns = [A0, A1], [W.Fn(W.F_ONE), W.Fn(W.F_ZPOW, 1)]
    p.region = W.Region(0.25, 0.5, 0.4, kind="points", points=np.array([0.0, 0.5], dtype=complex))
    p.U = W.probe(n, p.L, 5)
    both_paths(rs, p, lambda z: A0 + z * A1)
