"""The widest bands that the streaming solve takes and the next wider ones, in each
type: one launch more than the one-kernel solve (the block permutations) on this
side of the line, none beyond it, and on both sides the unrefined solutions'
normwise backward errors stay below 8 (2 kl + ku + 1) 2^-24 (2^-53 in FP64)."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

# n, kl, ku, real arithmetic, precision, streaming
LINE = [(700, 288, 288, False, 1, True), (700, 289, 288, False, 1, False), (640, 40, 536, False, 1, True),
        (900, 368, 368, False, 0, True), (900, 369, 368, False, 0, False),
        (2400, 2, 2350, True, 0, True), (2400, 3, 2350, True, 0, False),
        (2400, 2, 2270, True, 1, True), (2400, 3, 2270, True, 1, False)]


@pytest.mark.parametrize("n,kl,ku,real,precision,streams", LINE,
                         ids=["%s_%s_kl%d_ku%d" % ("real" if r else "complex", "mixed" if q else "fp64", a, b)
                              for _, a, b, r, q, _ in LINE])
def test_both_sides(n, kl, ku, real, precision, streams):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1605_07951_gb300 import rsrr
    p = W.random_banded(n=n, kl=kl, ku=ku, N=3, L=3, seed=n)
    if real:
        p.region = W.Region(0.5, 1.0, 0.1, kind="interval")
        p.U = np.asfortranarray(p.U.real.astype(np.complex128))
    launches = []
    for flags in (0, rsrr.RSRR_FLAG_PLAIN_SOLVE):
        s = rsrr.Solver(p, rsrr.default_opts(precision=precision, max_refine=0,
                                             flags=flags | (rsrr.RSRR_FLAG_REAL if real else 0)))
        s.sample()
        S = s.samples().copy()
        launches.append(s.stats()["launches"])
        z = s.points()
        s.close()
        rows = np.repeat(np.arange(n), np.diff(p.row_ptr))
        tol = 8.0 * (2 * kl + ku + 1) * (2.0 ** -53 if precision == 0 else 2.0 ** -24)
        for j in range(3):
            T = np.zeros((n, n), dtype=np.complex128)
            T[rows, p.col_idx] = p.values[0] + z[j] * p.values[1] + z[j] ** 2 * p.values[2]
            X = S[:, j * p.L:(j + 1) * p.L]
            r = np.abs(p.U - T @ X).max(axis=0)
            eta = r / (np.abs(T).sum(axis=1).max() * np.abs(X).max(axis=0) + np.abs(p.U).max(axis=0))
            assert eta.max() <= tol, (j, eta.max(), tol)
    assert launches[0] - launches[1] == (1 if streams else 0)
