"""What rsrr_zgemm keeps on the device between calls is at most 2 GiB, from the moment
the call returns (nothing synchronises in between) and also where the product
needed more than that."""
import ctypes

import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [500, 1500])
def test_bound_on_return(n):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1605_07951_gb300 import rsrr
    K = 40000
    A = torch.randn(n, K, dtype=torch.complex128, device="cuda")
    C = torch.empty(n, n, dtype=torch.complex128, device="cuda")

    def call(k):
        st = rsrr.rsrr_zgemm(n, n, k, 1, ctypes.c_void_p(A.data_ptr()), K, ctypes.c_void_p(A.data_ptr()), K,
                             ctypes.c_void_p(C.data_ptr()), n, 1.0, 0.0, rsrr.RSRR_GEMM_OZAKI, 1, 0, None)
        assert st == rsrr.RSRR_OK, rsrr.rsrr_last_error(None)

    call(16)  # the pool and the kernels are there
    rsrr.Solver(W.random_banded(n=20, kl=1, ku=1, N=1, L=1)).close()
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    call(K)
    kept = before - torch.cuda.mem_get_info()[0]
    assert 0 <= kept <= 2 << 30, kept
