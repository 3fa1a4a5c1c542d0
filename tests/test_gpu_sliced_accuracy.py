"""Rounding of long sliced products of few tiles, whose depth is split over the CTAs (32
splits here), on data of one sign, where no digit is lost to cancellation: the real
parts of A^H B with all components positive, against 80-bit or wider sums.

With u = 2^-53 and roundings of 0.41 u rms of the number rounded (uniform over a
binade), four chains of eight partial sums add (0.41 u)^2 8 / 12, their sum (0.41 u)^2
1.5, the partial sums' own roundings (0.41 u)^2 / 16: 0.61 u together, where one chain
of 32 has 1.34 u.  The bound of 0.9 u leaves half as much again to the sampling of 288
entries and to the depth's remainder."""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("method", [2, 3], ids=["tcgen05", "mma"])
@pytest.mark.parametrize("K", [20000, 33000, 40000])
def test_one_sign_sums(K, method):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1605_07951_gb300 import rsrr
    M, N = 12, 24
    rng = np.random.default_rng(K)
    A = np.abs(rng.standard_normal((M, K))) + 1j * np.abs(rng.standard_normal((M, K)))
    B = np.abs(rng.standard_normal((N, K))) + 1j * np.abs(rng.standard_normal((N, K)))
    dA, dB = torch.from_numpy(A).cuda(), torch.from_numpy(B).cuda()
    C = torch.empty(N, M, dtype=torch.complex128, device="cuda")
    st = rsrr.rsrr_zgemm(M, N, K, 1, ctypes.c_void_p(dA.data_ptr()), K, ctypes.c_void_p(dB.data_ptr()), K,
                         ctypes.c_void_p(C.data_ptr()), M, 1.0, 0.0, method, 0, 0, None)
    assert st == rsrr.RSRR_OK, rsrr.rsrr_last_error(None)
    got = C.cpu().numpy().T.real
    w = lambda x: x.astype(np.longdouble)
    ref = np.array([[(w(a.real) * w(b.real)).sum() + (w(a.imag) * w(b.imag)).sum() for b in B] for a in A])
    rel = ((w(got) - ref) / ref).astype(np.float64)
    assert np.sqrt((rel ** 2).mean()) <= 0.9 * 2.0 ** -53
