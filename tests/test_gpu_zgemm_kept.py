"""Device memory that rsrr_zgemm keeps between its calls is there for others: with
the rest of the device taken by an allocation of the test, a torch tensor, the
projection of a handle made before, and a request of a server made before get what
fits only without the kept memory, and give the same results as on a free device.
Products from several threads at once, with the kept memory given back meanwhile by
new handles, are the same bit for bit."""
import ctypes
import threading

import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

K, M = 40000, 500


@pytest.fixture(scope="module")
def env():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1605_07951_gb300 import rsrr
    A = torch.randn(M, K, dtype=torch.complex128, device="cuda")
    yield torch, rsrr, A
    del A
    torch.cuda.empty_cache()


def free(torch):
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    return torch.cuda.mem_get_info()[0]


def gram(env, n, C, stream=None):
    _, rsrr, A = env
    st = rsrr.rsrr_zgemm(n, n, K, 1, ctypes.c_void_p(A.data_ptr()), K, ctypes.c_void_p(A.data_ptr()), K,
                         ctypes.c_void_p(C.data_ptr()), n, 1.0, 0.0, rsrr.RSRR_GEMM_AUTO, 1, 0,
                         None if stream is None else ctypes.c_void_p(stream.cuda_stream))
    assert st == rsrr.RSRR_OK, rsrr.rsrr_last_error(None)


class Full:
    """After a product that keeps memory: all of the device but less than `need` bytes is
    taken, which the kept ones make up for."""

    def __init__(self, env, need):
        torch, rsrr, _ = env
        C = torch.empty(M, M, dtype=torch.complex128, device="cuda")
        rsrr.Solver(W.random_banded(n=40, kl=1, ku=1, N=1, L=1)).close()  # nothing is kept yet
        before = free(torch)
        gram(env, M, C)
        kept = before - free(torch)
        assert kept > 600 << 20 and need > 600 << 20, (kept, need)  # the sizes make the case
        self.torch, self.left = torch, need - min(need, kept) // 2

    def __enter__(self):
        self.rest = self.torch.empty(free(self.torch) - self.left, dtype=self.torch.uint8, device="cuda")
        assert free(self.torch) <= self.left + (4 << 20)

    def __exit__(self, *a):
        del self.rest
        self.torch.cuda.empty_cache()


def test_torch_beside_kept_memory(env):
    torch = env[0]
    with Full(env, 4 << 30):
        x = torch.empty(4 << 30, dtype=torch.uint8, device="cuda")
        del x


def problem():
    return W.rational_grid(g=120, N=16, L=40)


def test_projection_beside_kept_memory(env):
    torch, rsrr, _ = env
    twin = rsrr.Solver(problem())
    twin.sample()
    before = free(torch)
    twin.project()
    need = before - free(torch)
    P0 = twin.projected()
    twin.close()
    s = rsrr.Solver(problem())
    s.sample()
    with Full(env, need):
        s.project()
        P = s.projected()
    s.close()
    assert all(np.array_equal(a, b) for a, b in zip(P, P0))


def test_server_beside_kept_memory(env):
    torch, rsrr, _ = env
    sv = rsrr.Server(slots=1)
    before = free(torch)
    first = sv.wait(sv.submit(problem()))
    need = before - free(torch)
    sv.close()
    assert first["status"] in (rsrr.RSRR_OK, rsrr.RSRR_WGAP)
    sv = rsrr.Server(slots=1)
    with Full(env, need):
        r = sv.wait(sv.submit(problem()))
    sv.close()
    assert r["status"] == first["status"], r["error"]
    assert np.array_equal(r["lam"], first["lam"])


def test_threads_and_releases(env):
    torch, rsrr, _ = env
    sizes = [64, 130, 333, 500]
    ref = []
    for n in sizes:
        C = torch.empty(n, n, dtype=torch.complex128, device="cuda")
        gram(env, n, C)
        ref.append(C)
    stop, errors = threading.Event(), []

    def products(n, want):
        try:
            st = torch.cuda.Stream()
            C = torch.empty_like(want)
            for _ in range(12):
                C.fill_(float("nan"))
                torch.cuda.current_stream().synchronize()
                gram(env, n, C, st)
                if not torch.equal(C, want):
                    raise AssertionError(n)
        except BaseException as e:
            errors.append(e)

    def releases():
        try:
            p = W.random_banded(n=40, kl=1, ku=1, N=1, L=1)
            while not stop.is_set():
                rsrr.Solver(p).close()
        except BaseException as e:
            errors.append(e)

    ts = [threading.Thread(target=products, args=a) for a in zip(sizes, ref)]
    r = threading.Thread(target=releases)
    for t in ts + [r]:
        t.start()
    for t in ts:
        t.join()
    stop.set()
    r.join()
    assert not errors, errors
