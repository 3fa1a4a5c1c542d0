"""The work that users of the resolvent-sampling library have it do, as timed cases.

A case names an entry point (`call`) and its sizes:

  sample    rsrr_sample on a prepared handle, then rsrr_get_samples into a device
            tensor: the n x (N L) resolvent samples T(z_j)^{-1} U of one problem
  whole     rsrr_sample + rsrr_project + rsrr_solve: eigenvalues and eigenvectors
  band      rsrr_solve_band_noalloc: one banded system, no allocation
  gemm      rsrr_zgemm: one FP64-accurate complex product (a Gram matrix S^H S,
            a basis update R W)

Problem families (`family`): "grid", a rational NEP K - z M + z/(z - 300) E on a
g x h five-point grid (half-bandwidth g; the benchmark's is square, the whole
eigenproblems' are not, so that no two eigenvalues nearly coincide); "quadratic", a damped tridiagonal
quadratic NEP; "string", the loaded string at real Chebyshev points, in real
arithmetic; "sphere", the dense single-layer Helmholtz kernel on n points of the
unit sphere.  Sizes are those of the repository's benchmark, its request stream
and its tests, and what lies between them.
"""
import ctypes
import math

import numpy as np
import torch

from paper_1605_07951_gb300 import rsrr


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------
def listed():
    return [
        # a plug-in's single small banded system: launches and latency
        dict(name="band_n600", call="band", n=600, kl=7, ku=5, L=5),
        # a small damped quadratic problem, the smallest sampling request of a server
        dict(name="sample_quadratic_n1000", call="sample", family="quadratic", n=1000, N=32, L=8, fp64=False),
        # real points, real arithmetic: a loaded string on its interval of interest
        dict(name="sample_string_n400", call="sample", family="string", n=400, N=100, L=2, fp64=False),
        # a mid-size finite-element request of a server, default (mixed) precision
        dict(name="sample_grid_g61", call="sample", family="grid", g=61, h=61, N=32, L=16, fp64=False),
        # the same kind of request with the plain FP64 factorisation
        dict(name="sample_grid_g70_fp64", call="sample", family="grid", g=70, h=70, N=32, L=16, fp64=True),
        # the benchmark's problem: n = 40000, half-bandwidth 200, 64 points, 32 probes
        dict(name="sample_grid_g200", call="sample", family="grid", g=200, h=200, N=64, L=32, fp64=False),
        # a boundary-element request of a server (dense, ragged n)
        dict(name="sample_sphere_n500", call="sample", family="sphere", n=500, N=32, L=16, fp64=False),
        # a large boundary-element problem
        dict(name="sample_sphere_n2048", call="sample", family="sphere", n=2048, N=32, L=64, fp64=False),
        # the Gram matrix of a large basis
        dict(name="gram_40000x500", call="gemm", hermitian=True, M=500, N=500, K=40000),
        # a basis update: tall matrix times a small one
        dict(name="update_40000x237", call="gemm", hermitian=False, M=40000, N=237, K=237),
        # whole eigenproblems, sampling to eigenvectors: a server's request ...
        dict(name="whole_grid_g60", call="whole", family="grid", g=60, h=67, N=64, L=16, fp64=False),
        # ... and one of the benchmark's size
        dict(name="whole_grid_g200", call="whole", family="grid", g=200, h=187, N=64, L=32, fp64=False),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    call = rng.choice(["band", "sample", "sample", "sample", "sample", "gemm", "whole"])
    if call == "band":
        # every size drawn here fits the entry point's fixed work space
        return dict(call=call, n=_log_int(rng, 40, 6000), kl=rng.randint(1, 24), ku=rng.randint(1, 24),
                    L=rng.randint(1, 16))
    if call == "gemm":
        if rng.random() < 0.5:
            m = _log_int(rng, 24, 640)
            return dict(call=call, hermitian=True, M=m, N=m, K=_log_int(rng, 900, 60000))
        n = _log_int(rng, 24, 400)
        return dict(call=call, hermitian=False, M=_log_int(rng, 900, 60000), N=n, K=n)
    if call == "whole":
        g = _log_int(rng, 30, 140)
        return dict(call=call, family="grid", g=g, h=round(g * rng.uniform(1.06, 1.2)), N=rng.choice([32, 48, 64]),
                    L=rng.choice([12, 16, 24, 32]), fp64=False)
    family = rng.choice(["quadratic", "string", "grid", "grid", "grid", "sphere"])
    fp64 = rng.random() < 0.2
    if family == "quadratic":
        return dict(call=call, family=family, n=_log_int(rng, 200, 5000), N=rng.randint(8, 64),
                    L=rng.randint(1, 16), fp64=fp64)
    if family == "string":
        return dict(call=call, family=family, n=_log_int(rng, 100, 1500), N=rng.randint(12, 200),
                    L=rng.randint(1, 10), fp64=fp64)
    if family == "grid":
        g = _log_int(rng, 24, 100 if fp64 else 190)
        return dict(call=call, family=family, g=g, h=round(g * rng.uniform(0.8, 1.1)), N=rng.randint(8, 64),
                    L=rng.randint(1, 32), fp64=fp64)
    return dict(call=call, family=family, n=_log_int(rng, 100, 800 if fp64 else 2000), N=rng.randint(8, 32),
                L=rng.randint(4, 64), fp64=fp64)


# ---------------------------------------------------------------------------
# problem descriptions (what a user's program hands to rsrr.Solver)
# ---------------------------------------------------------------------------
class _Fn:
    def __init__(self, kind, param=0.0, scale=1.0):
        self.kind, self.param, self.scale = kind, param, scale


class _Region:
    def __init__(self, center, a, b, kind="ellipse"):
        self.center, self.a, self.b, self.kind = complex(center), float(a), float(b), kind


class _Problem:
    pass


def _probe(n, L, seed, real=False):
    """A complex normal probe matrix (the string's is real)."""
    rng = np.random.default_rng(seed)
    u = rng.standard_normal((L, n)) + (0.0 if real else 1j * rng.standard_normal((L, n)))
    return (u / np.sqrt(1.0 if real else 2.0)).astype(np.complex128).T  # column major


def _coo(case, seed):
    """n, rows, columns (sorted), the m value arrays, functions, region and half-bandwidth."""
    fam = case["family"]
    if fam == "grid":
        g, h = case["g"], case["h"]
        n, s = g * h, float((g + 1) ** 2)
        idx = np.arange(n)
        gi, gj = idx // g, idx % g
        rows, cols, kv = [idx], [idx], [np.full(n, 4.0 * s)]
        for di, dj in ((-1, 0), (0, -1), (0, 1), (1, 0)):
            ok = (gi + di >= 0) & (gi + di < h) & (gj + dj >= 0) & (gj + dj < g)
            rows.append(idx[ok])
            cols.append((idx + di * g + dj)[ok])
            kv.append(np.full(int(ok.sum()), -s))
        rows, cols, kv = np.concatenate(rows), np.concatenate(cols), np.concatenate(kv)
        order = np.lexsort((cols, rows))
        rows, cols, kv = rows[order], cols[order], kv[order]
        e = np.zeros(n)
        e[np.random.default_rng(seed).choice(n, size=round(0.01 * n), replace=False)] = 1.0
        diag = rows == cols
        vals = [kv, np.where(diag, 1.0, 0.0), np.where(diag, e[rows], 0.0)]
        fns = [_Fn(rsrr.RSRR_F_ONE), _Fn(rsrr.RSRR_F_ZPOW, 1, -1.0), _Fn(rsrr.RSRR_F_RATIONAL, 300.0)]
        return n, rows, cols, vals, fns, _Region(100.0, 80.0, 20.0), g
    n = case["n"]
    idx = np.arange(n)
    rows = np.concatenate([idx, idx[1:], idx[:-1]])
    cols = np.concatenate([idx, idx[1:] - 1, idx[:-1] + 1])
    order = np.lexsort((cols, rows))
    rows, cols = rows[order], cols[order]
    diag, last = rows == cols, (rows == n - 1) & (cols == n - 1)
    if fam == "quadratic":
        damping = np.random.default_rng(seed).uniform(0.0, 0.1, n)
        vals = [np.where(diag, 2.0 * n, -1.0 * n), np.where(diag, damping[rows], 0.0),
                np.where(diag, 4.0, 1.0) / (6.0 * n)]
        fns = [_Fn(rsrr.RSRR_F_ONE), _Fn(rsrr.RSRR_F_ZPOW, 1), _Fn(rsrr.RSRR_F_ZPOW, 2)]
        return n, rows, cols, vals, fns, _Region(-25.0 + 50.0j, 40.0, 40.0), 1
    # the loaded string: K_s + z/(z - 1) e_n e_n^T - z M at Chebyshev points of [3, 1e4]
    vals = [np.where(last, 1.0 * n, np.where(diag, 2.0 * n, -1.0 * n)), np.where(last, 1.0, 0.0),
            np.where(last, 2.0, np.where(diag, 4.0, 1.0)) / (6.0 * n)]
    fns = [_Fn(rsrr.RSRR_F_ONE), _Fn(rsrr.RSRR_F_RATIONAL, 1.0), _Fn(rsrr.RSRR_F_ZPOW, 1, -1.0)]
    return n, rows, cols, vals, fns, _Region(5001.5, 4998.5, 499.85, "interval"), 1


def _sphere(n, seed):
    """Quasi-uniform points (a Fibonacci lattice, seeded rotation) and the kernel's diagonal 1/(2h)."""
    i = np.arange(n) + 0.5
    phi, theta = np.arccos(1.0 - 2.0 * i / n), np.pi * (1.0 + 5.0 ** 0.5) * i
    P = np.stack([np.cos(theta) * np.sin(phi), np.sin(theta) * np.sin(phi), np.cos(phi)], axis=1)
    q, r = np.linalg.qr(np.random.default_rng(seed).standard_normal((3, 3)))
    P = np.ascontiguousarray(P @ (q * np.sign(np.diag(r))).T)
    d = np.linalg.norm(P[:, None, :] - P[None, :, :], axis=2) if n <= 1024 else None
    if d is not None:
        d[np.arange(n), np.arange(n)] = np.inf
        return P, 1.0 / (2.0 * d.min(axis=1).mean())
    near = []
    for s in range(0, n, 512):
        d = np.linalg.norm(P[s:s + 512, None, :] - P[None, :, :], axis=2)
        d[np.arange(d.shape[0]), np.arange(s, s + d.shape[0])] = np.inf
        near.append(d.min(axis=1))
    return P, 1.0 / (2.0 * np.concatenate(near).mean())


def _problem(case, seed):
    p = _Problem()
    p.N, p.L = case["N"], case["L"]
    if case["family"] == "sphere":
        p.n = case["n"]
        p.points, p.diag = _sphere(p.n, seed)
        p.region = _Region(3.0, 1.0, 1.0)
    else:
        p.n, rows, cols, p.values, p.fns, p.region, _ = _coo(case, seed)
        p.row_ptr = np.concatenate([[0], np.cumsum(np.bincount(rows, minlength=p.n))])
        p.col_idx = cols
    p.U = _probe(p.n, p.L, seed + 1, real=case["family"] == "string")
    return p


def _band_matrix(case, seed):
    """A diagonally weighted random band matrix in LAPACK's general band layout, and right-hand sides."""
    n, kl, ku, L = case["n"], min(case["kl"], case["n"] - 1), min(case["ku"], case["n"] - 1), case["L"]
    rng = np.random.default_rng(seed)
    ab = rng.standard_normal((kl + ku + 1, n)) + 1j * rng.standard_normal((kl + ku + 1, n))
    ab[ku] += 2.0 * (kl + ku)
    return n, kl, ku, np.asfortranarray(ab), _probe(n, L, seed + 1)


def _gemm_inputs(case, seed):
    """Matrices with columns of different sizes, as the columns of a sample matrix are."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    scale = torch.logspace(0, -6, case["K"] if not case["hermitian"] else case["M"], dtype=torch.float64, device="cuda")

    def normal(rows, cols):  # column major: cols x rows contiguous
        return torch.view_as_complex(torch.randn(cols, rows, 2, generator=gen, dtype=torch.float64, device="cuda"))

    if case["hermitian"]:
        A = normal(case["K"], case["M"]) * scale[:, None]
        return A, A
    return normal(case["M"], case["K"]) * scale[:, None], normal(case["K"], case["N"])


# ---------------------------------------------------------------------------
# a case: preparation, one pass
# ---------------------------------------------------------------------------
def prepare(case, seed):
    if case["call"] == "band":
        n, kl, ku, ab, U = _band_matrix(case, seed)
        return dict(case=case, n=n, kl=kl, ku=ku, L=case["L"], ab=torch.from_numpy(ab.T.copy()).cuda(),
                    U=torch.from_numpy(U.T.copy()).cuda(),
                    X=torch.empty(case["L"], n, dtype=torch.complex128, device="cuda"))
    if case["call"] == "gemm":
        A, B = _gemm_inputs(case, seed)
        return dict(case=case, A=A, B=B,
                    C=torch.empty(case["N"], case["M"], dtype=torch.complex128, device="cuda"))
    flags = rsrr.RSRR_FLAG_REAL if case["family"] == "string" else 0
    prec = rsrr.RSRR_PREC_FP64 if case["fp64"] else rsrr.RSRR_PREC_MIXED
    p = _problem(case, seed)
    solver = rsrr.Solver(p, rsrr.default_opts(precision=prec, flags=flags))
    state = dict(case=case, solver=solver, u0=p.U[:, 0].copy())
    if case["call"] == "sample":
        state["S"] = torch.empty(case["N"] * case["L"], p.n, dtype=torch.complex128, device="cuda")
    return state


def run(state):
    case = state["case"]
    if case["call"] == "band":
        st = rsrr.rsrr_solve_band_noalloc(state["n"], state["kl"], state["ku"], ctypes.c_void_p(state["ab"].data_ptr()),
                                          state["L"], ctypes.c_void_p(state["U"].data_ptr()),
                                          ctypes.c_void_p(state["X"].data_ptr()), None)
        if st != rsrr.RSRR_OK:
            raise RuntimeError(rsrr.rsrr_last_error(None).decode())
        return state["X"]
    if case["call"] == "gemm":
        A, B, C = state["A"], state["B"], state["C"]
        herm = int(case["hermitian"])
        st = rsrr.rsrr_zgemm(case["M"], case["N"], case["K"], herm, ctypes.c_void_p(A.data_ptr()), A.shape[1],
                             ctypes.c_void_p(B.data_ptr()), B.shape[1], ctypes.c_void_p(C.data_ptr()), case["M"],
                             1.0, 0.0, rsrr.RSRR_GEMM_AUTO, herm, 0, None)
        if st != rsrr.RSRR_OK:
            raise RuntimeError(rsrr.rsrr_last_error(None).decode())
        return C
    s = state["solver"]
    s.sample()
    if case["call"] == "sample":
        return s.samples(out=state["S"])
    s.project()
    out = s.solve()
    # an eigenvector's phase is free: the one in which its product with the first probe is positive
    V = out["V"]
    c = V.conj().T @ state["u0"]
    return dict(lam=out["lam"], V=V * (c / np.abs(c)))


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------
def work(case):
    if case["call"] == "band":
        n, kl, ku, L = case["n"], case["kl"], case["ku"], case["L"]
        return {"bytes": 16.0 * n * (kl + ku + 1 + 2 * L), "flops": 8.0 * n * (kl * ku + L * (2 * kl + ku))}
    if case["call"] == "gemm":
        M, N, K = case["M"], case["N"], case["K"]
        if case["hermitian"]:
            return {"bytes": 16.0 * (M * K + M * M), "flops": 4.0 * M * M * K}
        return {"bytes": 16.0 * (M * K + K * N + M * N), "flops": 8.0 * M * N * K}
    N, L = case["N"], case["L"]
    n = case["g"] * case["h"] if case["family"] == "grid" else case["n"]
    c = 2.0 if case["family"] == "string" else 8.0  # real or complex multiply-adds
    if case["family"] == "sphere":
        flops = N * (c * n ** 3 / 3 + c * n * n * L)
        reads = 24.0 * n
    else:
        w = case["g"] if case["family"] == "grid" else 1
        flops = N * (c * n * w * w + c * 2 * n * w * L)
        reads = 8.0 * 3 * (5 if case["family"] == "grid" else 3) * n
    samples = 16.0 * n * N * L
    if case["call"] == "sample":
        return {"bytes": reads + 16.0 * n * L + samples, "flops": flops}
    # the Gram matrix of the samples and one basis of half their number; the eigenvectors are few
    return {"bytes": reads + 16.0 * n * L + 16.0 * n * 32, "flops": flops + 4.0 * n * (N * L) ** 2}


# ---------------------------------------------------------------------------
# the same in plain torch, 64 bits
# ---------------------------------------------------------------------------
def _points(case):
    N = case["N"]
    if case["family"] == "string":
        return 5001.5 + 4998.5 * np.cos((2 * np.arange(N) + 1) * np.pi / (2 * N)) + 0j
    t = 2.0 * np.pi * (np.arange(N) + 0.5) / N
    center, a, b = {"grid": (100.0, 80.0, 20.0), "quadratic": (-25.0 + 50.0j, 40.0, 40.0),
                    "sphere": (3.0, 1.0, 1.0)}[case["family"]]
    return center + a * np.cos(t) + 1j * b * np.sin(t)


def _coefficients(family, z):
    if family == "grid":
        return [np.ones_like(z), -z, z / (z - 300.0)]
    if family == "quadratic":
        return [np.ones_like(z), z, z * z]
    return [np.ones_like(z), z / (z - 1.0), -z]


class _BlockTridiagonal:
    """Block LU of a batch of sparse banded matrices T_j = sum_i f_ij A_i (blocks at least the half-bandwidth)."""

    def __init__(self, n, rows, cols, vals, f, w, dev):
        b = max(w, 32)
        self.n, self.b, self.nb, self.N = n, b, -(-n // b), f[0].size
        t = sum(torch.as_tensor(fi, device=dev)[:, None] * torch.as_tensor(v, device=dev)[None, :] for fi, v in zip(f, vals))
        self.rows, self.cols, self.t = torch.as_tensor(rows, device=dev), torch.as_tensor(cols, device=dev), t
        start = np.searchsorted(rows, np.arange(0, self.nb + 1) * b)
        self.low, self.lu, self.up = [], [], []
        for k in range(self.nb):
            e = slice(start[k], start[k + 1])
            m = min(b, n - k * b)
            strip = torch.zeros(self.N, m, 3 * b, dtype=torch.complex128, device=dev)
            strip[:, self.rows[e] - k * b, self.cols[e] - (k - 1) * b] = t[:, e]
            lo, d, up = strip[:, :, :b], strip[:, :, b:b + m], strip[:, :, 2 * b:2 * b + max(0, min(b, n - (k + 1) * b))]
            if k:
                d = d - lo @ self.up[-1]
            lu, piv = torch.linalg.lu_factor(d)
            self.low.append(lo.clone())
            self.lu.append((lu, piv))
            self.up.append(torch.linalg.lu_solve(lu, piv, up) if up.shape[2] else up)

    def solve(self, R):  # (N, n, L)
        b, y = self.b, []
        for k in range(self.nb):
            r = R[:, k * b:(k + 1) * b]
            y.append(torch.linalg.lu_solve(*self.lu[k], r - self.low[k] @ y[-1] if k else r))
        for k in range(self.nb - 2, -1, -1):
            y[k] = y[k] - self.up[k] @ y[k + 1]
        return torch.cat(y, 1)

    def times(self, X):
        out = torch.zeros_like(X)
        for j in range(self.N):
            out[j].index_add_(0, self.rows, self.t[j][:, None] * X[j][self.cols])
        return out


def _solved(n, rows, cols, vals, f, w, U, dev):
    """X (N, n, L) = T_j^{-1} U, refined twice against the residual in 64 bits."""
    T = _BlockTridiagonal(n, rows, cols, vals, f, w, dev)
    B = torch.as_tensor(np.ascontiguousarray(U), device=dev)[None].expand(T.N, -1, -1)
    X = T.solve(B)
    for _ in range(2):
        X = X + T.solve(B - T.times(X))
    return X


def _eigenpairs(case, seed, dev):
    """The grid problem's real eigenvalues inside its ellipse: T(z) is real symmetric for real z."""
    n, rows, cols, vals, _, reg, _ = _coo(case, seed)
    K = torch.zeros(n, n, dtype=torch.float64, device=dev)
    r, c = torch.as_tensor(rows, device=dev), torch.as_tensor(cols, device=dev)
    K[r, c] = torch.as_tensor(vals[0], device=dev)
    e = torch.zeros(n, dtype=torch.float64, device=dev)
    e[r[r == c]] = torch.as_tensor(vals[2], device=dev)[r == c]
    start, vecs = torch.linalg.eigh(K + torch.diag(e * (100.0 / (100.0 - 300.0))))
    lam, V = [], []
    for i in range(n):
        l, v = float(start[i]), vecs[:, i].clone()
        if not 15.0 < l < 185.0:
            continue
        for _ in range(6):  # Newton on the Rayleigh functional, inverse iteration for the vector
            for _ in range(4):
                f, df = l / (l - 300.0), -300.0 / (l - 300.0) ** 2
                ve = float((v * v * e).sum())
                l -= (float(v @ (K @ v)) - l + f * ve) / (-1.0 + df * ve)
            T = K + torch.diag(e * (l / (l - 300.0)) - l * (1.0 + 1e-13))
            w = torch.linalg.solve(T, v[:, None])[:, 0]
            w = w / w.norm()
            done = float((w - v * torch.sign(w @ v)).norm()) < 1e-12
            v = w
            if done:
                break
        if abs(l - reg.center.real) < reg.a:
            lam.append(l)
            V.append(v)
    order = np.argsort(lam)
    lam = np.array(lam)[order] + 0j
    V = torch.stack(V, 1).cpu().numpy()[:, order].astype(np.complex128)
    c = V.conj().T @ _probe(n, case["L"], seed + 1)[:, 0]
    return dict(lam=lam, V=V * (c / np.abs(c)))


def exact(case, seed):
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    if case["call"] == "band":
        n, kl, ku, ab, U = _band_matrix(case, seed)
        j = np.concatenate([np.arange(max(0, -d), min(n, n - d)) for d in range(-ku, kl + 1)])  # columns of each diagonal
        d = np.concatenate([np.full(min(n, n - d) - max(0, -d), d) for d in range(-ku, kl + 1)])
        order = np.lexsort((j, j + d))
        j, d = j[order], d[order]
        X = _solved(n, j + d, j, [ab[ku + d, j]], [np.ones(1, np.complex128)], max(kl, ku), U, dev)
        return X[0].T.contiguous()
    if case["call"] == "gemm":
        A, B = _gemm_inputs(case, seed)  # columns are rows here: C^T = B^T op(A)^T
        return B @ A.conj().T if case["hermitian"] else B @ A
    if case["call"] == "whole":
        return _eigenpairs(case, seed, dev) if case["g"] * case["h"] <= 4500 else None
    z = _points(case)
    if case["family"] == "sphere":
        P, diag = _sphere(case["n"], seed)
        P = torch.as_tensor(P, device=dev)
        r = torch.linalg.norm(P[:, None, :] - P[None, :, :], dim=2)
        off = ~torch.eye(case["n"], dtype=torch.bool, device=dev)
        U = torch.as_tensor(np.ascontiguousarray(_probe(case["n"], case["L"], seed + 1)), device=dev)
        X = []
        for zj in z:
            T = torch.full(r.shape, complex(diag), dtype=torch.complex128, device=dev)
            T[off] = torch.exp(1j * complex(zj) * r[off]) / (4.0 * np.pi * r[off])
            X.append(torch.linalg.solve(T, U))
        X = torch.stack(X)
    else:
        n, rows, cols, vals, _, _, w = _coo(case, seed)
        U = _probe(n, case["L"], seed + 1, real=case["family"] == "string")
        X = _solved(n, rows, cols, vals, _coefficients(case["family"], z), w, U, dev)
    return X.transpose(1, 2).reshape(-1, X.shape[1])
