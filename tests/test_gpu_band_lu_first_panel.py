"""Clusters of the band LU whose work is over soon after they start: orders of one
to three panels, so that the first panel, which stores the row permutation into the
shared memory of the cluster's other CTAs, is most of a point, and more points than
clusters fit the GPU at once, so that CTAs start at all times.  The factors are those
of one CTA per point, bit for bit, whatever the size of the cluster (2 for narrow
upper parts, 8 for the widest here)."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", [3, 400])
@pytest.mark.parametrize("n,kl,ku", [(34, 33, 1), (35, 34, 34), (70, 40, 69), (96, 33, 95), (520, 70, 500)])
@pytest.mark.parametrize("precision", [0, 1], ids=["fp64", "mixed"])
def test_one_to_three_panels(n, kl, ku, N, precision):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1605_07951_gb300 import rsrr
    p = W.random_banded(n=n, kl=kl, ku=ku, N=N, L=2, seed=n)
    rows = np.repeat(np.arange(n), np.diff(p.row_ptr))
    p.values[0] = np.where(rows == p.col_idx, 0.05 * p.values[0], p.values[0])  # interchanges in most columns
    S = []
    for flags in (rsrr.RSRR_FLAG_ONE_CTA_LU, 0, 0):
        s = rsrr.Solver(p, rsrr.default_opts(precision=precision, max_refine=0, flags=flags))
        s.sample()
        S.append(s.samples().copy())
        s.close()
    assert np.isfinite(S[0]).all()
    assert np.array_equal(S[0], S[1]) and np.array_equal(S[0], S[2])
