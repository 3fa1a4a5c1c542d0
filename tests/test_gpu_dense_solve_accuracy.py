"""Rounding of the dense solve over many blocks: unrefined solutions of random matrices
with random right-hand sides, rms of the columns' normwise backward errors, computed
here in numpy.

A row of the right-hand sides takes n products.  Rounded by 0.41 u rms each, real and
imaginary parts of two products a term, one chain of all of them leaves about 0.41 u
sqrt(2 n / 2) x 1.4 = 0.58 sqrt(n) u in the forward and as much in the backward pass
(0.65 and 0.6 sqrt(n) u measured with one chain, n = 2048, in both precisions); sums
a block at a time leave sqrt(n / NB) roundings of the row and small ones, a fourth to
a sixth of that, beside the factor's own.  (Orders to 1024 sum by eights first.)  The bound of 0.4 sqrt(n) u lies between."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


class Terms:
    pass


@pytest.mark.parametrize("precision", [0, 1], ids=["fp64", "mixed"])
@pytest.mark.parametrize("n", [500, 1024, 1025, 1200, 2048])
def test_rounding_grows_by_blocks(n, precision):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1605_07951_gb300 import rsrr
    rng = np.random.default_rng(n)
    p = Terms()
    p.n, p.N, p.L = n, 4, 24
    p.As = [rng.standard_normal((n, n)) + 1j * rng.standard_normal((n, n)) for _ in range(2)]
    p.fns = [W.Fn(W.F_ONE), W.Fn(W.F_ZPOW, 1)]
    p.region = W.Region(0.1, 0.5, 0.4)
    p.U = W.probe(n, p.L, 3)
    s = rsrr.Solver(p, rsrr.default_opts(precision=precision, max_refine=0))
    s.sample()
    S, z = s.samples().copy(), s.points()
    s.close()
    eta = []
    for j in range(p.N):
        T, X = p.As[0] + z[j] * p.As[1], S[:, j * p.L:(j + 1) * p.L]
        r = np.abs(p.U - T @ X).max(axis=0)
        eta.append(r / (np.abs(T).sum(axis=1).max() * np.abs(X).max(axis=0) + np.abs(p.U).max(axis=0)))
    u = 2.0 ** -53 if precision == 0 else 2.0 ** -24
    assert np.sqrt(np.mean(np.square(eta))) <= 0.4 * np.sqrt(n) * u
