"""The estimate of a handle's device bytes follows the sizes of what it holds.  With one
sampling point it is smooth in the number of probe columns L where no operand of a
product grows by a tile: the buffers are quadratic in L with small factors, the
inverses of SS-FULL's 16 nodes come in blocks of 16 rows (0.3 MB), so second
differences over L stay below 4 MiB.  FP64 products, which do without operand slices,
ask for less than sliced ones where those are large."""
import numpy as np
import pytest

import workloads as W
from paper_1605_07951_gb300 import rsrr as rs


def estimate(n, N, L, gemm):
    p = W.quadratic_tridiag(n=n, N=N, L=1)
    return rs.estimate_bytes(p, rs.default_opts(gemm=gemm, NQ=16), L=L)


@pytest.mark.parametrize("gemm,L0,L1", [(rs.RSRR_GEMM_FP64, 60, 71), (rs.RSRR_GEMM_AUTO, 34, 65),
                                        (rs.RSRR_GEMM_OZAKI, 34, 65)], ids=["fp64", "auto", "sliced"])
@pytest.mark.parametrize("n", [3000, 20000])
def test_smooth_in_L(n, gemm, L0, L1):
    b = np.array([estimate(n, 1, L, gemm) for L in range(L0, L1)], dtype=np.int64)
    assert np.abs(np.diff(b, 2)).max() <= 4 << 20, np.diff(b, 2)


@pytest.mark.parametrize("n,N,L", [(9000, 4, 65), (20000, 16, 16), (20000, 1, 64)])
def test_fp64_products_ask_for_less(n, N, L):
    fp64 = estimate(n, N, L, rs.RSRR_GEMM_FP64)
    assert all(fp64 + (32 << 20) < estimate(n, N, L, g) for g in (rs.RSRR_GEMM_AUTO, rs.RSRR_GEMM_OZAKI))
