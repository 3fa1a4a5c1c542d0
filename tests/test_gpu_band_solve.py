"""Streaming band solve at the edges of its shapes: half-bandwidths around the
32-row groups that choose the rows and columns a lane updates, point and probe
counts that choose 2, 4, 8 or 16 right-hand sides per CTA (ragged last chunks),
n off the block size, and interchanges that lengthen the rows of U.

The unrefined solutions' normwise backward errors, computed here in numpy, stay
below 8 (2 kl + ku + 1) 2^-24 (2^-53 for FP64), as for the band LU; every shape
does the same operations on a column, so the first right-hand sides of the first
points have the same bits whatever N and L are."""
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


@pytest.mark.parametrize("precision", [0, 1], ids=["fp64", "mixed"])
@pytest.mark.parametrize("n,kl,ku", [(70, 1, 1), (333, 31, 33), (330, 64, 65), (400, 96, 97), (500, 128, 120),
                                     (520, 160, 161), (700, 200, 224), (800, 250, 257)])
def test_every_shape(rs, n, kl, ku, precision):
    p = W.random_banded(n=n, kl=kl, ku=ku, N=64, L=33, seed=n)
    rows = np.repeat(np.arange(n), np.diff(p.row_ptr))
    p.values[0] = np.where(rows == p.col_idx, 0.05 * p.values[0], p.values[0])
    z = oracle.sample_points(p.region, p.N)
    tol = 8.0 * (2 * kl + ku + 1) * (2.0 ** -53 if precision == 0 else 2.0 ** -24)
    first = None
    U = p.U
    for N, L in ((64, 33), (20, 33), (10, 18), (3, 2)):  # 16, 8, 4, 2 right-hand sides per CTA in complex64
        p.region = W.Region(p.region.center, p.region.a, p.region.b, kind="points", points=z[:N])
        p.U = np.asfortranarray(U[:, :L])
        s = rs.Solver(p, rs.default_opts(precision=precision, max_refine=0), N=N, L=L)
        s.sample()
        S = s.samples()
        s.close()
        head = np.stack([S[:, j * L:j * L + 2] for j in range(3)])
        if first is None:
            first = head
        assert np.array_equal(head, first), (N, L)
        for j in (0, 1, N - 1):
            T = np.zeros((n, n), dtype=np.complex128)
            T[rows, p.col_idx] = p.values[0] + z[j] * p.values[1] + z[j] ** 2 * p.values[2]
            X = S[:, j * L:(j + 1) * L]
            r = np.abs(p.U - T @ X).max(axis=0)
            eta = r / (np.abs(T).sum(axis=1).max() * np.abs(X).max(axis=0) + np.abs(p.U).max(axis=0))
            assert eta.max() <= tol, (N, L, j, eta.max(), tol)
