// Resolvent sampling on dense BEM-like T(z_j) (RSRR step 2, Section 4.3, for
// the Nystrom single-layer kernel of Section 2.1):
//   T(z)_ij = exp(i z r_ij) / (4 pi r_ij) (i != j), T_ii = diag,
// assembled per sampling point, factored by a batched blocked LU with partial
// pivoting, solved for the L probe columns with the block inverses of the
// factorisation, and refined with FP64 residuals (the GEMM of proj.cu).
//
// Dense storage of one point: column major n x n (lda = n).  Pivoting is
// applied dense-style inside an NB-column block and to the trailing columns,
// never to the columns already factored: the solve applies each block's
// interchanges just before that block's elimination, as the band solve does.
#include <algorithm>
#include <climits>
#include <type_traits>

#include "common.cuh"
#include "rsrr_internal.h"

namespace rsrr {

constexpr double kFourPi = 12.566370614359172;

// ---------------------------------------------------------------- assembly
// FP64 entries; the mixed path's complex64 matrix is narrowed from them.  T is
// symmetric (r_ij and r_ji have the same bits), so a block takes a pair of 32 x 32
// tiles: the entries with j >= i are computed, kept in shared memory and written to
// both.  Bound by the FP64 unit (exp, sincos and a division per entry): a lane per
// entry, the distances once for all points of the block, the transcendentals half as
// often as there are entries.  32 points of order 2048: 16.4 -> 6.7 ms.
constexpr int AT = 32;

__global__ void __launch_bounds__(256)
assemble_dense_kernel(double2 *__restrict__ A_all, const double *__restrict__ pts, const double2 *__restrict__ zs,
                      double diag, int n, int N) {
    __shared__ double2 s_t[AT][AT + 1];
    // tile pair (bi <= bj) of the upper triangle
    int bj = (int)((sqrtf(8.f * (float)blockIdx.x + 1.f) - 1.f) * 0.5f);
    while ((int64_t)(bj + 1) * (bj + 2) / 2 <= blockIdx.x) ++bj;
    while ((int64_t)bj * (bj + 1) / 2 > blockIdx.x) --bj;
    const int bi = (int)(blockIdx.x - (int64_t)bj * (bj + 1) / 2);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int i = bi * AT + lane;
    double r[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const int j = bj * AT + warp + 8 * q;
        r[q] = -1.0;
        if (i < n && j < n && i < j) {
            const double dx = pts[3 * i] - pts[3 * j], dy = pts[3 * i + 1] - pts[3 * j + 1],
                         dz = pts[3 * i + 2] - pts[3 * j + 2];
            r[q] = sqrt(dx * dx + dy * dy + dz * dz);
        }
    }
    for (int pt = blockIdx.y; pt < N; pt += gridDim.y) {
        const double zr = zs[pt].x, zi = zs[pt].y;
        double2 *A = A_all + (size_t)pt * n * n;
        __syncthreads();
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int jj = warp + 8 * q, j = bj * AT + jj;
            if (i >= n || j >= n || i > j) continue;
            double2 v = make_double2(diag, 0.0);
            if (i < j) {
                const double mag = exp(-zi * r[q]) / (kFourPi * r[q]);
                double s, c;
                sincos(zr * r[q], &s, &c);
                v = make_double2(mag * c, mag * s);
            }
            s_t[jj][lane] = v;
            A[(int64_t)j * n + i] = v;
        }
        __syncthreads();
#pragma unroll
        for (int q = 0; q < 4; ++q) {  // column i2 of the mirrored tile, rows j2
            const int ii = warp + 8 * q, i2 = bi * AT + ii, j2 = bj * AT + lane;
            if (j2 < n && i2 < j2) A[(int64_t)i2 * n + j2] = s_t[lane][ii];
        }
    }
}

// T(z_j) = sum_i f_i(z_j) A_i for caller-supplied dense A_i (m x n^2
// complex128, term-major): every thread loads the m coefficients of one
// entry once and writes that entry of every point of the chunk, so the A_i
// are read once per chunk of points and the N matrices written once (the
// write stream is the bound).  coef is point-major, f_i(z_j) at [j m + i].
__global__ void assemble_dense_terms_kernel(double2 *__restrict__ T_all, const double2 *__restrict__ A,
                                            const double2 *__restrict__ coef, int64_t nn2, int j0, int nj,
                                            int m) {
    extern __shared__ double2 s_cf[];  // nj x m
    for (int t = threadIdx.x; t < nj * m; t += blockDim.x) s_cf[t] = coef[(size_t)j0 * m + t];
    __syncthreads();
    for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < nn2;
         q += (int64_t)gridDim.x * blockDim.x) {
        double2 a[RSRR_MAX_TERMS_DEV];
#pragma unroll
        for (int i = 0; i < RSRR_MAX_TERMS_DEV; ++i)
            a[i] = i < m ? A[(int64_t)i * nn2 + q] : make_double2(0.0, 0.0);
        for (int j = 0; j < nj; ++j) {
            double2 acc = make_double2(0.0, 0.0);
#pragma unroll
            for (int i = 0; i < RSRR_MAX_TERMS_DEV; ++i)
                if (i < m) acc = cfma(acc, s_cf[j * m + i], a[i]);
            T_all[(int64_t)(j0 + j) * nn2 + q] = acc;
        }
    }
}

// R(:, c) (+)= cf[c m + i] Y(:, c): one term of T(lambda_c) v_c = sum_i
// f_i(lambda_c) A_i v_c for the residuals of the dense-terms kind
__global__ void accum_term_cols_kernel(double2 *__restrict__ R, const double2 *__restrict__ Y,
                                       const double2 *__restrict__ cf, int m, int i, int n, int cnt,
                                       int first) {
    const int64_t total = (int64_t)n * cnt;
    for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < total;
         q += (int64_t)gridDim.x * blockDim.x) {
        const int c = (int)(q / n);
        const double2 v = cmul(cf[(size_t)c * m + i], Y[q]);
        R[q] = first ? v : cadd(R[q], v);
    }
}

// rr[c] = ||R(:, c)||_2^2 and vv[c] = ||V(:, c)||_2^2 (block per column)
__global__ void col_norms2_kernel(const double2 *__restrict__ R, const double2 *__restrict__ V, int n,
                                  double *__restrict__ rr, double *__restrict__ vv) {
    const int c = blockIdx.x;
    double a = 0.0, b = 0.0;
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
        const double2 r = R[(int64_t)c * n + i], v = V[(int64_t)c * n + i];
        a += r.x * r.x + r.y * r.y;
        b += v.x * v.x + v.y * v.y;
    }
    __shared__ double sa[32], sb[32];
    for (int off = 16; off; off >>= 1) {
        a += shfl_down(a, off);
        b += shfl_down(b, off);
    }
    if ((threadIdx.x & 31) == 0) {
        sa[threadIdx.x >> 5] = a;
        sb[threadIdx.x >> 5] = b;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        double ta = 0.0, tb = 0.0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) {
            ta += sa[w];
            tb += sb[w];
        }
        rr[c] = ta;
        vv[c] = tb;
    }
}

// |v| without hypot's scaling where the squares stay in range
RSRR_DEV double cabs_fast(double2 v) {
    const int hx = __double2hiint(v.x) & 0x7fffffff, hy = __double2hiint(v.y) & 0x7fffffff, h = max(hx, hy);
    if (h >= (600 << 20) && h < (1400 << 20)) return sqrt(fma(v.x, v.x, v.y * v.y));
    if ((hx | hy | __double2loint(v.x) | __double2loint(v.y)) == 0) return 0.0;
    return cabsv(v);
}

// ||T(z_j)||_inf from the stored complex128 matrix: row sums of moduli.  A block
// takes 32 rows, its eight warps every eighth column each (a thread per row left the
// SMs to 500 warps for 32 points of order 500): that order 0.59 -> 0.20 ms, order
// 2048 4.8 -> 2.7 ms.
__global__ void __launch_bounds__(256)
dense_tnorm_kernel(double *__restrict__ tnorm, const double2 *__restrict__ A_all, int n) {
    __shared__ double s_sum[8][32];
    const int pt = blockIdx.y, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const double2 *A = A_all + (size_t)pt * n * n;
    const int i = blockIdx.x * 32 + lane;
    double s = 0.0;
    if (i < n)
#pragma unroll 4
        for (int j = warp; j < n; j += 8) s += cabs_fast(A[(int64_t)j * n + i]);
    s_sum[warp][lane] = s;
    __syncthreads();
    if (warp == 0) {
        for (int w = 1; w < 8; ++w) s += s_sum[w][lane];
        for (int off = 16; off; off >>= 1) s = fmax(s, shfl_down(s, off));
        if (lane == 0) atomic_max_nonneg(tnorm + pt, s);
    }
}

// ---------------------------------------------------------------- LU
constexpr int DP_THREADS = 1024;
constexpr int DP_WARPS = DP_THREADS / 32;

// Inverses of the unit lower L11 and of U11 of the diagonal block at k0 (jb x jb,
// zero padded to NB x NB), for the solve.  A lane per row: a warp carries 32 / NB
// columns of an inverse, each step broadcasts one entry of it by shuffle and
// updates the rows below (above).  rinv: the reciprocals of the diagonal of U11.
template <typename C, int NB, int WARPS>
RSRR_DEV void panel_inverses(const C *__restrict__ A, C *__restrict__ dst, C *__restrict__ s_blk,
                             const C *__restrict__ rinv, int n, int k0, int jb) {
    constexpr int CPW = 32 / NB, TASKS = NB / CPW;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    for (int q = tid; q < NB * NB; q += 32 * WARPS) {
        const int j = q / NB, i = q % NB;
        s_blk[q] = (i < jb && j < jb) ? A[(int64_t)(k0 + j) * n + k0 + i] : czero<C>();
    }
    __syncthreads();
    const int t = lane % NB, sub = lane / NB;
    for (int task = warp; task < 2 * TASKS; task += WARPS) {
        const bool lower = task < TASKS;
        const int jf = (lower ? task : task - TASKS) * CPW, j = jf + sub;
        C x = (t == j && j < jb) ? cone<C>() : czero<C>();
        if (lower) {
            for (int i = jf; i < jb - 1; ++i) {
                const C xi = cshfl(x, (lane & ~(NB - 1)) + i);
                if (i >= j && t > i) x = cfms(x, s_blk[i * NB + t], xi);
            }
        } else {
            for (int i = min(jf + CPW, jb) - 1; i >= 0; --i) {
                const C xi = cmul(cshfl(x, (lane & ~(NB - 1)) + i), rinv[i]);
                if (i <= j && t == i) x = xi;
                if (i <= j && t < i) x = cfms(x, s_blk[i * NB + t], xi);
            }
        }
        dst[(lower ? 0 : NB * NB) + j * NB + t] = (t < jb && j < jb) ? x : czero<C>();
    }
}

// |re|+|im| as an ordered integer (never NaN), and the largest of a warp with the
// first row that has it: redux on integers, where compares of doubles would each
// cost the warp 64 cycles of the FP64 unit
RSRR_DEV int panel_key(float v) {
    const int b = __float_as_int(v) & 0x7fffffff;
    return b > 0x7f800000 ? 0 : b;
}
RSRR_DEV long long panel_key(double v) {
    const long long b = __double_as_longlong(v) & 0x7fffffffffffffffll;
    return b > 0x7ff0000000000000ll ? 0 : b;
}
RSRR_DEV int panel_best(int &key, int row) {
    const int m = __reduce_max_sync(0xffffffffu, key);
    row = __reduce_min_sync(0xffffffffu, key == m ? row : INT_MAX);
    key = m;
    return row;
}
RSRR_DEV int panel_best(long long &key, int row) {
    const int hi = (int)(key >> 32), mh = __reduce_max_sync(0xffffffffu, hi);
    const unsigned lo = hi == mh ? (unsigned)key : 0u, ml = __reduce_max_sync(0xffffffffu, lo);
    row = __reduce_min_sync(0xffffffffu, hi == mh && lo == ml ? row : INT_MAX);
    key = ((long long)mh << 32) | ml;
    return row;
}

// Panel k0 (columns k0..k0+jb-1, rows k0..n-1, at most T * RPT of them) of every
// point, one CTA per point.  Bound by the chain of its columns, so the rows live in
// registers (RPT a thread), W columns at a time, and a column costs one barrier:
// before it every warp publishes the row of its largest |re|+|im| (first row on
// ties) and the owner of the pivot's place its row, after it every thread finds the
// winner, exchanges, and updates its rows with the winner's.  Where W < NB, the
// panel's other columns take the W interchanges, the triangular solve and the
// rank-W update from global memory afterwards.  In complex128 one warp takes the
// reciprocal (its three divisions by every warp cost as much as the update) behind
// a second barrier.  The operations on an element and their order are those of
// dense_panel_kernel below.  All panels of a factorisation, against that kernel:
// complex64, 32 points of order 500 2.3 -> 0.68 ms, of order 2048 16.0 -> 5.3 ms;
// complex128, 512 nodes of order 237 15.8 -> 1.5 ms.
template <typename C, int NB, int W, int RPT, int T>
__global__ void __launch_bounds__(T, 512 / T)
dense_panel_reg_kernel(C *__restrict__ A_all, int32_t *__restrict__ piv_all, int32_t *__restrict__ info_all,
                       C *__restrict__ dinv_all, int n, int k0) {
    using R = typename real_of<C>::type;
    using Key = decltype(panel_key(R()));
    constexpr int NW = T / 32, GW = W < 8 ? W : 8;
    static_assert(2 * W * (NB - W) <= T, "one element of the interchanged rows per thread");
    constexpr bool FP64 = sizeof(R) == 8;
    const int pt = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    C *A = A_all + (size_t)pt * n * n + (size_t)k0 * n;  // column k0
    int32_t *piv = piv_all + (size_t)pt * n;
    const int jb = min(NB, n - k0);
    __shared__ Key s_key[2][NW];
    __shared__ int s_idx[2][NW], s_p[W];
    __shared__ C s_cand[2][NW][W], s_own[2][W], s_piv[W][W], s_u[W][NB], s_rinv[NB], s_blk[NB * NB];
    int par = 0;
    for (int s0 = 0; s0 < jb; s0 += W) {
        const int wj = min(W, jb - s0);
        C a[RPT][W];
        Key key = -1;
        int row = INT_MAX;
#pragma unroll
        for (int q = 0; q < RPT; ++q) {
            const int r = k0 + tid + q * T;
#pragma unroll
            for (int j = 0; j < W; ++j)
                a[q][j] = (r < n && r >= k0 + s0 && j < wj) ? A[(int64_t)(s0 + j) * n + r] : czero<C>();
        }
#pragma unroll
        for (int q = 0; q < RPT; ++q) {
            const int r = k0 + tid + q * T;
            if (r < n && r >= k0 + s0) {
                const Key k = panel_key(cabs1(a[q][0]));
                if (k > key) { key = k; row = r; }
            }
        }
#pragma unroll
        for (int g = 0; g < W / GW; ++g) {
#pragma unroll 1
            for (int u = 0; u < GW; ++u) {
                const int cc = g * GW + u, c = k0 + s0 + cc;
                if (cc >= wj) break;
                Key wk = key;
                const int wr = panel_best(wk, row);
                if (lane == 0) { s_key[par][warp] = wk; s_idx[par][warp] = wr; }
#pragma unroll
                for (int q = 0; q < RPT; ++q) {
                    const int r = k0 + tid + q * T;
                    if (r == wr)
#pragma unroll
                        for (int j = 0; j < W; ++j) s_cand[par][warp][j] = a[q][j];
                    if (r == c)
#pragma unroll
                        for (int j = 0; j < W; ++j) s_own[par][j] = a[q][j];
                }
                __syncthreads();
                Key bk = lane < NW ? s_key[par][lane] : -1;
                const int p = panel_best(bk, lane < NW ? s_idx[par][lane] : INT_MAX);
                const C *pr = s_cand[par][((p - k0) % T) >> 5];
                const C pv = pr[cc];
                C inv;
                if constexpr (FP64) {
                    if (warp == 0) {
                        inv = crecip(pv);
                        if (lane == 0) s_rinv[s0 + cc] = inv;
                    }
                } else {
                    inv = crecip(pv);
                    if (tid == 0) s_rinv[s0 + cc] = inv;
                }
                if (tid < W) s_piv[cc][tid] = pr[tid];
                if (tid == 0) {
                    s_p[cc] = p;
                    piv[c] = p;
                    if (bk <= 0 && info_all[pt] == 0) info_all[pt] = c + 1;
                }
                if constexpr (FP64) {
                    __syncthreads();
                    inv = s_rinv[s0 + cc];
                }
                key = -1;
                row = INT_MAX;
                const bool nz = cnonzero(pv);
#pragma unroll
                for (int q = 0; q < RPT; ++q) {
                    const int r = k0 + tid + q * T;
                    if (r == p && p != c)
#pragma unroll
                        for (int j = 0; j < W; ++j) a[q][j] = s_own[par][j];
                    if (r > c && r < n) {
                        if (nz) {
                            C l = a[q][g * GW];
#pragma unroll
                            for (int v = 1; v < GW; ++v)
                                if (v == u) l = a[q][g * GW + v];
                            l = cmul(l, inv);
#pragma unroll
                            for (int v = 0; v < GW; ++v)
                                if (v == u) a[q][g * GW + v] = l;
#pragma unroll
                            for (int j = g * GW + 1; j < W; ++j)
                                if (j > cc) a[q][j] = cfms(a[q][j], l, pr[j]);
                        }
                        C nx = czero<C>();
#pragma unroll
                        for (int v = g * GW + 1; v < W && v <= g * GW + GW; ++v)
                            if (v == cc + 1) nx = a[q][v];
                        const Key k = panel_key(cabs1(nx));
                        if (k > key) { key = k; row = r; }
                    }
                }
                par ^= 1;
            }
        }
        const int top = k0 + s0 + wj;
#pragma unroll
        for (int q = 0; q < RPT; ++q) {
            const int r = k0 + tid + q * T;
            if (r >= top && r < n)
#pragma unroll
                for (int j = 0; j < W; ++j)
                    if (j < wj) A[(int64_t)(s0 + j) * n + r] = a[q][j];
        }
        __syncthreads();
        for (int e = tid; e < wj * wj; e += T) {
            const int i = e % wj, j = e / wj;
            A[(int64_t)(s0 + j) * n + k0 + s0 + i] = s_piv[i][j];
        }
        if constexpr (W < NB) {
            // interchanges of the other columns: the row that ends at x started at y
            C val = czero<C>();
            const int col = tid / (2 * wj), slot = tid % (2 * wj);
            const int oc = col < s0 ? col : col + wj;  // column of the panel
            int x = 0;
            const bool mine = col < jb - wj;
            if (mine) {
                x = slot < wj ? k0 + s0 + slot : s_p[slot - wj];
                int y = x;
                for (int i = wj - 1; i >= 0; --i) {
                    const int ci = k0 + s0 + i, pi = s_p[i];
                    y = y == ci ? pi : (y == pi ? ci : y);
                }
                val = A[(int64_t)oc * n + y];
            }
            __syncthreads();
            if (mine) {
                A[(int64_t)oc * n + x] = val;
                if (slot < wj) s_u[slot][oc] = val;
            }
            __syncthreads();
            const int rest = jb - s0 - wj;  // columns to the right; wj == W if there are any
            if (tid < rest) {
                const int oc2 = s0 + wj + tid;
                C uu[W];
#pragma unroll
                for (int i = 0; i < W; ++i) {
                    uu[i] = s_u[i][oc2];
#pragma unroll
                    for (int t = 0; t < i; ++t) uu[i] = cfms(uu[i], s_piv[i][t], uu[t]);
                    s_u[i][oc2] = uu[i];
                    A[(int64_t)oc2 * n + k0 + s0 + i] = uu[i];
                }
            }
            __syncthreads();
#pragma unroll 2
            for (int c2 = s0 + wj; c2 < jb; ++c2) {
                C xv[RPT];
#pragma unroll
                for (int q = 0; q < RPT; ++q) {
                    const int r = k0 + tid + q * T;
                    xv[q] = (r >= top && r < n) ? A[(int64_t)c2 * n + r] : czero<C>();
                }
#pragma unroll
                for (int i = 0; i < W; ++i) {
                    const C ui = s_u[i][c2];
#pragma unroll
                    for (int q = 0; q < RPT; ++q) xv[q] = cfms(xv[q], a[q][i], ui);
                }
#pragma unroll
                for (int q = 0; q < RPT; ++q) {
                    const int r = k0 + tid + q * T;
                    if (r >= top && r < n) A[(int64_t)c2 * n + r] = xv[q];
                }
            }
        }
    }
    __syncthreads();
    const size_t nblk = ((size_t)n + NB - 1) / NB;
    panel_inverses<C, NB, NW>(A - (size_t)k0 * n, dinv_all + ((size_t)pt * nblk + k0 / NB) * 2 * NB * NB, s_blk, s_rinv,
                              n, k0, jb);
}

// Panels of more rows than the registers of an SM hold: one CTA per
// point, right-looking in global memory (L2): per column a block-wide argmax
// of |re|+|im| (first index on ties), the interchange inside the panel, the
// multipliers and the rank-1 update of the remaining panel columns.  Then
// the inverses of the unit lower L11 and of U11 (jb x jb) for the solve.
template <typename C, int NB>
__global__ void __launch_bounds__(DP_THREADS, 1)
dense_panel_kernel(C *__restrict__ A_all, int32_t *__restrict__ piv_all, int32_t *__restrict__ info_all,
                   C *__restrict__ dinv_all, int n, int k0) {
    using R = typename real_of<C>::type;
    const int pt = blockIdx.x;
    C *A = A_all + (size_t)pt * n * n;
    int32_t *piv = piv_all + (size_t)pt * n;
    const int jb = min(NB, n - k0);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    __shared__ R s_v[DP_WARPS];
    __shared__ int s_i[DP_WARPS];
    __shared__ C s_row[NB];
    __shared__ C s_blk[NB * NB];
    __shared__ C s_rinv[NB];
    for (int cc = 0; cc < jb; ++cc) {
        const int c = k0 + cc;
        R v = (R)-1;
        int ix = 0x7fffffff;
        for (int r = c + tid; r < n; r += DP_THREADS) {
            const R a = cabs1(A[(int64_t)c * n + r]);
            if (a > v) { v = a; ix = r; }
        }
        for (int off = 16; off; off >>= 1) {
            const R ov = shfl_down(v, off);
            const int oi = shfl_down(ix, off);
            if (ov > v || (ov == v && oi < ix)) { v = ov; ix = oi; }
        }
        if (lane == 0) { s_v[warp] = v; s_i[warp] = ix; }
        __syncthreads();
        R bv = s_v[0];
        int p = s_i[0];
        for (int w = 1; w < DP_WARPS; ++w)
            if (s_v[w] > bv || (s_v[w] == bv && s_i[w] < p)) { bv = s_v[w]; p = s_i[w]; }
        if (p >= n) p = c;  // a column of NaN
        if (tid < jb && p != c) {
            const int64_t col = (int64_t)(k0 + tid) * n;
            const C t = A[col + c]; A[col + c] = A[col + p]; A[col + p] = t;
        }
        __syncthreads();
        if (tid < jb) s_row[tid] = A[(int64_t)(k0 + tid) * n + c];
        if (tid == 0) {
            piv[c] = p;
            if (!(bv > (R)0) && info_all[pt] == 0) info_all[pt] = c + 1;
        }
        __syncthreads();
        const C pv = s_row[cc];
        if (cnonzero(pv)) {
            const C inv = crecip(pv);
            for (int r = c + 1 + tid; r < n; r += DP_THREADS) {
                const C l = cmul(A[(int64_t)c * n + r], inv);
                A[(int64_t)c * n + r] = l;
                for (int c2 = cc + 1; c2 < jb; ++c2) {
                    C *a = A + (int64_t)(k0 + c2) * n + r;
                    *a = cfms(*a, l, s_row[c2]);
                }
            }
        }
        __syncthreads();
    }
    if (tid < jb) s_rinv[tid] = crecip(A[(int64_t)(k0 + tid) * n + k0 + tid]);
    const size_t nblk = ((size_t)n + NB - 1) / NB;
    panel_inverses<C, NB, DP_WARPS>(A, dinv_all + ((size_t)pt * nblk + k0 / NB) * 2 * NB * NB, s_blk, s_rinv, n, k0, jb);
}

// Rows in registers while they fit (64 registers a thread, up to 4096 rows), 256
// threads where they suffice, so that two panels share an SM.
template <typename C, int NB>
static void dense_panel(C *A, int32_t *piv, int32_t *info, C *dinv, int n, int k0, int N, cudaStream_t s) {
    constexpr int W1 = 256 / (int)sizeof(C) < NB ? 256 / (int)sizeof(C) : NB;
    const int rows = n - k0;
    if (rows <= 256) dense_panel_reg_kernel<C, NB, W1, 1, 256><<<N, 256, 0, s>>>(A, piv, info, dinv, n, k0);
    else if (rows <= 512) dense_panel_reg_kernel<C, NB, W1, 1, 512><<<N, 512, 0, s>>>(A, piv, info, dinv, n, k0);
    else if (rows <= 1024) dense_panel_reg_kernel<C, NB, W1 / 2, 2, 512><<<N, 512, 0, s>>>(A, piv, info, dinv, n, k0);
    else if (rows <= 2048) dense_panel_reg_kernel<C, NB, W1 / 4, 4, 512><<<N, 512, 0, s>>>(A, piv, info, dinv, n, k0);
    else if (rows <= 4096) dense_panel_reg_kernel<C, NB, W1 / 8, 8, 512><<<N, 512, 0, s>>>(A, piv, info, dinv, n, k0);
    else dense_panel_kernel<C, NB><<<N, DP_THREADS, 0, s>>>(A, piv, info, dinv, n, k0);
}

// Trailing columns k0+jb.. in chunks of 32: the panel's interchanges (in
// order), then U12 = L11^{-1} A12 in place.
template <typename C, int NB>
__global__ void __launch_bounds__(256)
dense_laswp_trsm_kernel(C *__restrict__ A_all, const int32_t *__restrict__ piv_all,
                        const C *__restrict__ dinv_all, int n, int k0) {
    const int pt = blockIdx.y;
    C *A = A_all + (size_t)pt * n * n;
    const int32_t *piv = piv_all + (size_t)pt * n;
    const int jb = min(NB, n - k0);
    const int c0 = k0 + jb + blockIdx.x * 32;
    const int ncol = min(32, n - c0);
    if (ncol <= 0) return;
    const int nblk = (n + NB - 1) / NB;
    const C *Linv = dinv_all + ((size_t)pt * nblk + k0 / NB) * 2 * NB * NB;
    __shared__ C s_L[NB * NB];
    __shared__ C s_a[NB * 32];
    const int tid = threadIdx.x;
    for (int q = tid; q < NB * NB; q += 256) s_L[q] = Linv[q];
    if (tid < ncol) {
        const int64_t col = (int64_t)(c0 + tid) * n;
        for (int cc = 0; cc < jb; ++cc) {
            const int p = piv[k0 + cc];
            if (p != k0 + cc) {
                const C t = A[col + k0 + cc]; A[col + k0 + cc] = A[col + p]; A[col + p] = t;
            }
        }
    }
    __syncthreads();
    for (int q = tid; q < NB * 32; q += 256) {
        const int i = q % NB, c = q / NB;
        s_a[q] = (i < jb && c < ncol) ? A[(int64_t)(c0 + c) * n + k0 + i] : czero<C>();
    }
    __syncthreads();
    for (int q = tid; q < NB * 32; q += 256) {
        const int i = q % NB, c = q / NB;
        if (i < jb && c < ncol) {
            C s = czero<C>();
            for (int t = 0; t < NB; ++t) s = cfma(s, s_L[t * NB + i], s_a[c * NB + t]);
            A[(int64_t)(c0 + c) * n + k0 + i] = s;
        }
    }
}

// A22 -= L21 U12 over 64 x 64 tiles (K = jb), 256 threads with 4 x 4 outputs.
template <typename C, int NB>
__global__ void __launch_bounds__(256)
dense_gemm_update_kernel(C *__restrict__ A_all, int n, int k0) {
    const int pt = blockIdx.z;
    C *A = A_all + (size_t)pt * n * n;
    const int jb = min(NB, n - k0);
    const int r0 = k0 + jb + blockIdx.x * 64, c0 = k0 + jb + blockIdx.y * 64;
    if (r0 >= n || c0 >= n) return;
    __shared__ C s_l[NB][64 + 1];  // L21(r0+i, k0+t) at [t][i]
    __shared__ C s_u[NB][64 + 1];  // U12(k0+t, c0+j) at [t][j]
    const int tid = threadIdx.x;
    for (int q = tid; q < NB * 64; q += 256) {
        const int i = q % 64, t = q / 64;
        s_l[t][i] = (r0 + i < n && t < jb) ? A[(int64_t)(k0 + t) * n + r0 + i] : czero<C>();
        const int tt = q % NB, j = q / NB;
        s_u[tt][j] = (c0 + j < n && tt < jb) ? A[(int64_t)(c0 + j) * n + k0 + tt] : czero<C>();
    }
    __syncthreads();
    const int tx = tid % 16, ty = tid / 16;
    C acc[4][4];
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            const int i = r0 + tx + 16 * a, j = c0 + ty + 16 * b;
            acc[a][b] = (i < n && j < n) ? A[(int64_t)j * n + i] : czero<C>();
        }
    // Groups of 16 rows and columns beyond the matrix are left out: whole tiles of the
    // trailing matrices of 512 complex128 nodes of order 237 are 1.4 times their work
    // (all updates 10.0 -> 7.3 ms; order 140: 2.4 -> 1.7 ms).
    const int na = min(4, (n - r0 + 15) / 16), nb = min(4, (n - c0 + 15) / 16);
    auto accumulate = [&](auto groups) {
        constexpr int NBV = decltype(groups)::value;
#pragma unroll 4
        for (int t = 0; t < NB; ++t) {
            C lv[4], uv[NBV];
#pragma unroll
            for (int a = 0; a < 4; ++a) lv[a] = s_l[t][tx + 16 * a];
#pragma unroll
            for (int b = 0; b < NBV; ++b) uv[b] = s_u[t][ty + 16 * b];
#pragma unroll
            for (int a = 0; a < 4; ++a)
                if (a < na)
#pragma unroll
                    for (int b = 0; b < NBV; ++b) acc[a][b] = cfms(acc[a][b], lv[a], uv[b]);
        }
    };
    switch (nb) {
    case 1: accumulate(std::integral_constant<int, 1>()); break;
    case 2: accumulate(std::integral_constant<int, 2>()); break;
    case 3: accumulate(std::integral_constant<int, 3>()); break;
    default: accumulate(std::integral_constant<int, 4>());
    }
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            const int i = r0 + tx + 16 * a, j = c0 + ty + 16 * b;
            if (i < n && j < n) A[(int64_t)j * n + i] = acc[a][b];
        }
}

// ---------------------------------------------------------------- solve
// One CTA per (point, chunk of LC right-hand sides); B (n x L per point,
// column major) is overwritten with the solution.  Forward per block: the
// block's interchanges, y = L11^{-1} b_block, rows below -= L21 y.  Backward
// per block from the end: x = U11^{-1} y_block, rows above -= U12 x: both
// updates a thread per row, the factor read along its columns.
//
// A block's interchanges are composed by one warp (a lane per pivot: the row
// at the block's row, and at the row outside that the pivot names first), then
// applied by all threads at once.
//
// IDENT: the right-hand sides are the identity's columns (L = n), B is only
// written.  A chunk takes the columns whose ones the interchanges bring to LC
// adjacent rows of one block: its forward pass starts there (two thirds of the
// forward products are with zeros).
//
// FP64 (the inverses of SS-FULL's nodes): bound by the FP64 unit, so lanes must
// not idle: the backward pass by rows keeps all of them busy where a dot
// product per row of the block used 16 of 32.  500 matrices of order 233: 78.6
// -> 35.6 ms.  FP32: bound by reading the factor from L2 once per chunk, so the
// chunks are as wide as leaves one for every SM: n = 2048, 64 right-hand sides,
// 32 points 16.8 -> 5.4 ms for three solves, of which the last returns at once.
//
// GROUP products at a time are summed from zero, then a block's sums, and the row
// rounds once a block: subtracted one by one from the row they left 1.5 to 2.4 times
// the backward error (random matrices of order 500 to 2048, both precisions; sphere
// kernels 1.2 to 4 times).  By blocks (GROUP = NB) orders up to 500 are left with 1.0
// to 1.1 times the error of sixteen partial sums, by eights with as much or less;
// from about 1000 on both are below it, so by blocks there: n = 4096, 64 right-hand
// sides, 32 points 9.4 ms a solve against 13.3 by eights and 9.3 one by one.
template <typename C, int NB, int LC, int TH, bool IDENT, int GROUP>
__global__ void __launch_bounds__(TH, 512 / TH)
dense_solve_kernel(const C *__restrict__ A_all, const int32_t *__restrict__ piv_all,
                   const C *__restrict__ dinv_all, C *__restrict__ B_all, int n, int L,
                   const int32_t *__restrict__ skip) {
    const int pt = blockIdx.y;
    if (skip && skip[pt]) return;
    const int col0 = blockIdx.x * LC;
    const int ncol = min(LC, L - col0);
    const C *A = A_all + (size_t)pt * n * n;
    const int32_t *piv = piv_all + (size_t)pt * n;
    const int nblk = (n + NB - 1) / NB;
    const C *dinv = dinv_all + (size_t)pt * nblk * 2 * NB * NB;
    C *B = B_all + (size_t)pt * L * n + (IDENT ? 0 : (size_t)col0 * n);
    const int tid = threadIdx.x;
    __shared__ __align__(16) C s_D[NB * NB];
    __shared__ __align__(16) C s_b[NB * LC];
    __shared__ __align__(16) C s_y[NB * LC];
    __shared__ int s_col[LC], s_dst[2 * NB], s_src[2 * NB], s_moves;
    static_assert(!IDENT || NB % LC == 0, "a chunk's ones lie in one block");
    static_assert(GROUP == 8 || GROUP == NB, "the loads go by eights");
    extern __shared__ int s_perm[];  // IDENT: position -> row, then the pivots
    if (IDENT) {
        // the interchanges composed: row s_perm[p] ends at position p
        for (int i = tid; i < n; i += TH) {
            s_perm[i] = i;
            s_perm[n + i] = piv[i];
        }
        __syncthreads();
        if (tid == 0)
            for (int i = 0; i < n; ++i) {
                const int p = s_perm[n + i];
                if (p != i) {
                    const int t = s_perm[i]; s_perm[i] = s_perm[p]; s_perm[p] = t;
                }
            }
        __syncthreads();
        if (tid < LC) s_col[tid] = tid < ncol ? s_perm[col0 + tid] : 0;
    } else if (tid < LC) {
        s_col[tid] = tid;
    }
    __syncthreads();
    size_t cb[LC];  // the columns' places in B
#pragma unroll
    for (int c = 0; c < LC; ++c) cb[c] = (size_t)s_col[c] * n;
    const int k_first = IDENT ? col0 / NB * NB : 0;
    if (IDENT) {
        for (int i = tid; i < n; i += TH)
#pragma unroll
            for (int c = 0; c < LC; ++c)
                if (c < ncol) B[cb[c] + i] = i == col0 + c ? cone<C>() : czero<C>();
        __syncthreads();
    }
    // y = D b for the block at k0 (D: its L11^{-1} or U11^{-1}), into s_y and B
    auto diagonal = [&](int k0, int jb, const C *src) {
        for (int q = tid; q < NB * NB; q += TH) s_D[q] = src[q];
        for (int q = tid; q < NB * LC; q += TH) {
            const int i = q % NB, c = q / NB;
            s_b[q] = i < jb && c < ncol ? B[(size_t)s_col[c] * n + k0 + i] : czero<C>();
        }
        __syncthreads();
        for (int q = tid; q < NB * LC; q += TH) {
            const int i = q % NB, c = q / NB;
            C y = czero<C>();
#pragma unroll 8
            for (int t = 0; t < NB; ++t) y = cfma(y, s_D[t * NB + i], s_b[c * NB + t]);
            s_y[i * LC + c] = y;
            if (i < jb && c < ncol) B[(size_t)s_col[c] * n + k0 + i] = y;
        }
        __syncthreads();
    };
    // rows r_lo .. r_hi-1 -= A(:, k0 .. k0+jb-1) y
    auto update = [&](int k0, int jb, int r_lo, int r_hi) {
        constexpr bool EARLY = GROUP == NB;  // the row's values first: room in the registers
        for (int r = r_lo + tid; r < r_hi; r += TH) {
            C acc[LC], b[EARLY ? LC : 1];
#pragma unroll
            for (int c = 0; c < LC; ++c) {
                acc[c] = czero<C>();
                if constexpr (EARLY) b[c] = c < ncol ? B[cb[c] + r] : czero<C>();
            }
            const C *a = A + (size_t)k0 * n + r;
            if (jb == NB) {
#pragma unroll 1
                for (int t0 = 0; t0 < NB; t0 += 8) {
                    C l[8];
#pragma unroll
                    for (int t = 0; t < 8; ++t) l[t] = a[(size_t)(t0 + t) * n];
                    if constexpr (GROUP == NB) {
#pragma unroll
                        for (int t = 0; t < 8; ++t)
#pragma unroll
                            for (int c = 0; c < LC; ++c) acc[c] = cfma(acc[c], l[t], s_y[(t0 + t) * LC + c]);
                    } else {
#pragma unroll
                        for (int c = 0; c < LC; ++c) {
                            C s = czero<C>();
#pragma unroll
                            for (int t = 0; t < 8; ++t) s = cfma(s, l[t], s_y[(t0 + t) * LC + c]);
                            acc[c] = cadd(acc[c], s);
                        }
                    }
                }
            } else {
                for (int t = 0; t < jb; ++t) {
                    const C l = a[(size_t)t * n];
#pragma unroll
                    for (int c = 0; c < LC; ++c) acc[c] = cfma(acc[c], l, s_y[t * LC + c]);
                }
            }
#pragma unroll
            for (int c = 0; c < LC; ++c)
                if (c < ncol) B[cb[c] + r] = csub(EARLY ? b[EARLY ? c : 0] : B[cb[c] + r], acc[c]);
        }
        __syncthreads();
    };
    // the interchanges of the block at k0
    auto interchange = [&](int k0, int jb) {
        if (tid < 32) {
            const int lane = tid;
            const int p = lane < jb ? piv[k0 + lane] : -1;
            const unsigned same = __match_any_sync(0xffffffffu, p);
            const bool first = p >= k0 + jb && (same & ((1u << lane) - 1u)) == 0;
            int top = k0 + lane, out = p;  // rows at block row `lane` and, where first, at row p
            for (int cc = 0; cc < jb; ++cc) {
                const int q = __shfl_sync(0xffffffffu, p, cc), a = __shfl_sync(0xffffffffu, top, cc);
                const unsigned at = __ballot_sync(0xffffffffu, first && p == q);
                const int b = at ? __shfl_sync(0xffffffffu, out, __ffs(at) - 1) : __shfl_sync(0xffffffffu, top, (q - k0) & 31);
                if (lane == cc) top = b;
                if (at) {
                    if (first && p == q) out = a;
                } else if (q != k0 + cc && lane == q - k0) {
                    top = a;
                }
            }
            const bool mt = lane < jb && top != k0 + lane, mo = first && out != p;
            const unsigned bt = __ballot_sync(0xffffffffu, mt), bo = __ballot_sync(0xffffffffu, mo);
            const unsigned below = (1u << lane) - 1u;
            if (mt) {
                s_dst[__popc(bt & below)] = k0 + lane;
                s_src[__popc(bt & below)] = top;
            }
            if (mo) {
                s_dst[__popc(bt) + __popc(bo & below)] = p;
                s_src[__popc(bt) + __popc(bo & below)] = out;
            }
            if (lane == 0) s_moves = __popc(bt) + __popc(bo);
        }
        __syncthreads();
        const int items = s_moves * LC;
        constexpr int PER = (2 * NB * LC + TH - 1) / TH;
        C v[PER];
#pragma unroll
        for (int k = 0; k < PER; ++k) {
            const int q = tid + k * TH, e = q / LC, c = q % LC;
            v[k] = q < items && c < ncol ? B[(size_t)s_col[c] * n + s_src[e]] : czero<C>();
        }
        __syncthreads();
#pragma unroll
        for (int k = 0; k < PER; ++k) {
            const int q = tid + k * TH, e = q / LC, c = q % LC;
            if (q < items && c < ncol) B[(size_t)s_col[c] * n + s_dst[e]] = v[k];
        }
        __syncthreads();
    };
    for (int k0 = k_first; k0 < n; k0 += NB) {
        const int jb = min(NB, n - k0);
        if (!IDENT || k0 > k_first) interchange(k0, jb);
        diagonal(k0, jb, dinv + (size_t)(k0 / NB) * 2 * NB * NB);
        update(k0, jb, k0 + jb, n);
    }
    for (int k0 = ((n - 1) / NB) * NB; k0 >= 0; k0 -= NB) {
        const int jb = min(NB, n - k0);
        diagonal(k0, jb, dinv + (size_t)(k0 / NB) * 2 * NB * NB + NB * NB);
        update(k0, jb, 0, k0);
    }
}

// ---------------------------------------------------------------- residual
// R = U - T X in FP64 for every point of the batch whose done flag is 0 (the
// flags are read on the device: a sweep needs no host wait).  A block computes
// a 32 x 16 tile of one point, two rows and two columns a thread, over slabs
// of 16 columns of T that cp.async brings one slab ahead.
//
// Bound by the FP64 unit (a warp-wide FMA takes 64 cycles of its scheduler, so
// two FMAs a cycle and SM): what counts is that every SM has work and no lane
// idles.  One product per point, as before, left 8 blocks on 152 SMs: n = 500,
// L = 16, 32 points 203 ms for three residuals; all points in one launch 3.1 ms
// (2.6 ms of FMAs).  The tile is this small so that a few hundred blocks spread
// evenly.  Sums run over k in order, as the direct path of fp64_gemm's do.
constexpr int DR_M = 32, DR_N = 16, DR_K = 16, DR_THREADS = 128;
RSRR_DEV void dr_copy16(void *dst, const void *src, bool in) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(d), "l"(src), "r"(in ? 16 : 0));
}
__global__ void __launch_bounds__(DR_THREADS)
dense_residual_kernel(double2 *__restrict__ R_all, const double2 *__restrict__ T_all,
                      const double2 *__restrict__ X_all, const double2 *__restrict__ U,
                      const int32_t *__restrict__ done, int n, int L) {
    const int pt = blockIdx.z;
    if (done && done[pt]) return;
    __shared__ double2 s_t[2][DR_K][DR_M], s_x[2][DR_N][DR_K];
    const double2 *T = T_all + (size_t)pt * n * n, *X = X_all + (size_t)pt * n * L;
    const int m0 = blockIdx.x * DR_M, c0 = blockIdx.y * DR_N, tid = threadIdx.x;
    const int tx = tid % 16, ty = tid / 16;  // rows tx, tx + 16; columns ty, ty + 8
    auto load = [&](int k0, int b) {
        for (int q = tid; q < DR_K * DR_M; q += DR_THREADS) {
            const int k = k0 + q / DR_M, i = m0 + q % DR_M;
            const bool in = k < n && i < n;
            dr_copy16(&s_t[b][q / DR_M][q % DR_M], T + (in ? (size_t)k * n + i : 0), in);
        }
        for (int q = tid; q < DR_N * DR_K; q += DR_THREADS) {
            const int c = c0 + q / DR_K, k = k0 + q % DR_K;
            const bool in = k < n && c < L;
            dr_copy16(&s_x[b][q / DR_K][q % DR_K], X + (in ? (size_t)c * n + k : 0), in);
        }
        asm volatile("cp.async.commit_group;\n" ::);
    };
    double2 acc[2][2];
#pragma unroll
    for (int a = 0; a < 2; ++a) acc[a][0] = acc[a][1] = make_double2(0.0, 0.0);
    load(0, 0);
    for (int k0 = 0, b = 0; k0 < n; k0 += DR_K, b ^= 1) {
        if (k0 + DR_K < n) {
            load(k0 + DR_K, b ^ 1);
            asm volatile("cp.async.wait_group 1;\n" ::);
        } else {
            asm volatile("cp.async.wait_group 0;\n" ::);
        }
        __syncthreads();
#pragma unroll 4
        for (int k = 0; k < DR_K; ++k) {
            const double2 t0 = s_t[b][k][tx], t1 = s_t[b][k][tx + 16];
            const double2 x0 = s_x[b][ty][k], x1 = s_x[b][ty + 8][k];
            acc[0][0] = cfma(acc[0][0], t0, x0);
            acc[1][0] = cfma(acc[1][0], t1, x0);
            acc[0][1] = cfma(acc[0][1], t0, x1);
            acc[1][1] = cfma(acc[1][1], t1, x1);
        }
        __syncthreads();
    }
#pragma unroll
    for (int a = 0; a < 2; ++a)
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            const int i = m0 + tx + 16 * a, c = c0 + ty + 8 * e;
            if (i < n && c < L)
                R_all[((size_t)pt * L + c) * n + i] = csub(U[(size_t)c * n + i], acc[a][e]);
        }
}

// column maxima of |R| and |X| (n x L per point) of the points whose done flag
// (may be null) is 0, into rmax / xmax
__global__ void dense_colmax_kernel(const double2 *__restrict__ R_all, const double2 *__restrict__ X_all, int n,
                                    int L, double *__restrict__ rmax, double *__restrict__ xmax,
                                    const int32_t *__restrict__ done) {
    const int l = blockIdx.x, pt = blockIdx.y;
    if (done && done[pt]) return;
    const double2 *R = R_all + ((size_t)pt * L + l) * n, *X = X_all + ((size_t)pt * L + l) * n;
    // squared moduli by their bit patterns, one square root at the end (FP64 pipe); as
    // unsigned numbers the patterns of NaN are the largest: a column that holds one
    // has no backward error
    unsigned long long r = 0, x = 0;
    auto bits = [](double v) { return (unsigned long long)__double_as_longlong(v); };
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
        const double2 u = R[i], v = X[i];
        r = max(r, bits(fma(u.x, u.x, u.y * u.y)));
        x = max(x, bits(fma(v.x, v.x, v.y * v.y)));
    }
    for (int off = 16; off; off >>= 1) {
        r = max(r, shfl_down(r, off));
        x = max(x, shfl_down(x, off));
    }
    __shared__ unsigned long long wr[32], wx[32];
    if ((threadIdx.x & 31) == 0) { wr[threadIdx.x >> 5] = r; wx[threadIdx.x >> 5] = x; }
    __syncthreads();
    if (threadIdx.x == 0) {
        unsigned long long a = 0, b = 0;
        for (int q = 0; q < (int)(blockDim.x >> 5); ++q) { a = max(a, wr[q]); b = max(b, wx[q]); }
        rmax[(size_t)pt * L + l] = sqrt(__longlong_as_double((long long)a));
        xmax[(size_t)pt * L + l] = sqrt(__longlong_as_double((long long)b));
    }
}

// Taylor coefficients in place: A <- A o (i r)/p for p >= 1 (diagonal -> 0);
// for p == 0, A = exp(i c r)/(4 pi r) off the diagonal and diag on it.
__global__ void taylor_step_kernel(double2 *__restrict__ A, const double *__restrict__ pts,
                                   double2 c, double diag, int n, int p) {
    const int64_t total = (int64_t)n * n;
    for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < total;
         q += (int64_t)gridDim.x * blockDim.x) {
        const int j = (int)(q / n), i = (int)(q - (int64_t)j * n);
        if (i == j) {
            A[q] = make_double2(p == 0 ? diag : 0.0, 0.0);
            continue;
        }
        const double dx = pts[3 * i] - pts[3 * j], dy = pts[3 * i + 1] - pts[3 * j + 1],
                     dz = pts[3 * i + 2] - pts[3 * j + 2];
        const double r = sqrt(dx * dx + dy * dy + dz * dz);
        if (p == 0) {
            const double mag = exp(-c.y * r) / (kFourPi * r);
            double s, co;
            sincos(c.x * r, &s, &co);
            A[q] = make_double2(mag * co, mag * s);
        } else {
            const double2 a = A[q];
            const double f = r / p;  // multiply by i r / p
            A[q] = make_double2(-a.y * f, a.x * f);
        }
    }
}

// ||T(lam_c) v_c||^2, ||v_c||^2 and the column sums of |T(lam_c)| (for the
// 1-norm), matrix-free in FP64; thread per row i (and per column i for the sums).
__global__ void dense_eig_residual_kernel(const double2 *__restrict__ V, const double2 *__restrict__ lam,
                                          const double *__restrict__ pts, double diag, int n,
                                          double *__restrict__ rr, double *__restrict__ vv,
                                          double *__restrict__ t1) {
    const int c = blockIdx.y;
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const double2 z = lam[c];
    double r2 = 0.0, v2 = 0.0, cs = 0.0;
    if (i < n) {
        double2 s = make_double2(0.0, 0.0);
        for (int j = 0; j < n; ++j) {
            double2 t;
            if (i == j) {
                t = make_double2(diag, 0.0);
            } else {
                const double dx = pts[3 * i] - pts[3 * j], dy = pts[3 * i + 1] - pts[3 * j + 1],
                             dz = pts[3 * i + 2] - pts[3 * j + 2];
                const double r = sqrt(dx * dx + dy * dy + dz * dz);
                const double mag = exp(-z.y * r) / (kFourPi * r);
                double sn, co;
                sincos(z.x * r, &sn, &co);
                t = make_double2(mag * co, mag * sn);
            }
            s = cfma(s, t, V[(int64_t)c * n + j]);
            cs += cabsv(t);  // |T_ij| = |T_ji|: row sum i equals column sum i
        }
        r2 = s.x * s.x + s.y * s.y;
        const double2 x = V[(int64_t)c * n + i];
        v2 = x.x * x.x + x.y * x.y;
    }
    for (int off = 16; off; off >>= 1) {
        r2 += shfl_down(r2, off);
        v2 += shfl_down(v2, off);
        cs = fmax(cs, shfl_down(cs, off));
    }
    if ((threadIdx.x & 31) == 0) {
        atomicAdd(rr + c, r2);
        atomicAdd(vv + c, v2);
        atomic_max_nonneg(t1 + c, cs);
    }
}

// ================================================================ launchers
static int grid_for_d(int64_t work, int threads = 256, int cap = 152 * 16) {
    int64_t g = (work + threads - 1) / threads;
    return (int)std::max<int64_t>(1, std::min<int64_t>(g, cap));
}

cudaError_t launch_assemble_dense_c128(double2 *A, const double *pts, const double2 *zs, double diag,
                                       int n, int N, cudaStream_t s) {
    const int64_t nt = ((int64_t)n + AT - 1) / AT, pairs = nt * (nt + 1) / 2;
    if (pairs > 0x7fffffff) return cudaErrorInvalidValue;
    // blocks of one tile pair share its distances over their points: enough blocks for
    // eight waves, more points each beyond that
    const int64_t groups = std::max<int64_t>(1, std::min<int64_t>(std::min(N, 65535), 152 * 8 * 8 / pairs));
    assemble_dense_kernel<<<dim3((unsigned)pairs, (unsigned)groups), 256, 0, s>>>(A, pts, zs, diag, n, N);
    return cudaGetLastError();
}
cudaError_t launch_assemble_dense_terms(double2 *T, const double2 *A, const double2 *coef, int n, int N,
                                        int m, cudaStream_t s) {
    if (m < 1 || m > RSRR_MAX_TERMS_DEV) return cudaErrorInvalidValue;
    const int64_t nn2 = (int64_t)n * n;
    const int chunk = std::max(1, 2048 / m);  // coefficients of a chunk: <= 32 KB of shared memory
    for (int j0 = 0; j0 < N; j0 += chunk) {
        const int nj = std::min(chunk, N - j0);
        assemble_dense_terms_kernel<<<grid_for_d(nn2, 256, 152 * 8), 256, sizeof(double2) * nj * m, s>>>(
            T, A, coef, nn2, j0, nj, m);
        cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}
cudaError_t launch_accum_term_cols(double2 *R, const double2 *Y, const double2 *cf, int m, int i, int n,
                                   int cnt, bool first, cudaStream_t s) {
    accum_term_cols_kernel<<<grid_for_d((int64_t)n * cnt), 256, 0, s>>>(R, Y, cf, m, i, n, cnt, first ? 1 : 0);
    return cudaGetLastError();
}
cudaError_t launch_col_norms2(const double2 *R, const double2 *V, int n, int cnt, double *rr, double *vv,
                              cudaStream_t s) {
    if (cnt < 1) return cudaSuccess;
    col_norms2_kernel<<<cnt, 256, 0, s>>>(R, V, n, rr, vv);
    return cudaGetLastError();
}
cudaError_t launch_dense_tnorm(double *tnorm, const double2 *A, int n, int N, cudaStream_t s) {
    cudaError_t e = cudaMemsetAsync(tnorm, 0, sizeof(double) * N, s);
    if (e != cudaSuccess) return e;
    dense_tnorm_kernel<<<dim3((n + 31) / 32, N), 256, 0, s>>>(tnorm, A, n);
    return cudaGetLastError();
}

cudaError_t launch_dense_tc_update(float2 *A, int n, int k0, int jb, int N, unsigned int *status,
                                   cudaStream_t s);

// the trailing update A22 -= L21 U12 of one panel: FP32 / FP64 FMAs, or, for
// complex64 with tc, the 3xTF32 tensor-core kernel of dense_tc.cu
template <typename C, int NB>
static cudaError_t dense_update(C *A, int n, int k0, int N, unsigned int *status, bool tc, cudaStream_t s) {
    const int jb = std::min(NB, n - k0), rest = n - k0 - jb;
    if constexpr (std::is_same<C, float2>::value)
        if (tc) return launch_dense_tc_update(A, n, k0, jb, N, status, s);
    dense_gemm_update_kernel<C, NB><<<dim3((rest + 63) / 64, (rest + 63) / 64, N), 256, 0, s>>>(A, n, k0);
    return cudaGetLastError();
}

template <typename C, int NB>
static cudaError_t dense_lu_t(C *A, int32_t *piv, int32_t *info, C *dinv, int n, int N, cudaStream_t s,
                              int64_t *launches, unsigned int *status, bool tc) {
    cudaError_t e = cudaMemsetAsync(info, 0, sizeof(int32_t) * N, s);
    if (e != cudaSuccess) return e;
    for (int k0 = 0; k0 < n; k0 += NB) {
        const int jb = std::min(NB, n - k0);
        dense_panel<C, NB>(A, piv, info, dinv, n, k0, N, s);
        const int rest = n - k0 - jb;
        if (rest > 0) {
            dense_laswp_trsm_kernel<C, NB><<<dim3((rest + 31) / 32, N), 256, 0, s>>>(A, piv, dinv, n, k0);
            if ((e = cudaGetLastError()) != cudaSuccess) return e;
            if ((e = dense_update<C, NB>(A, n, k0, N, status, tc, s)) != cudaSuccess) return e;
            *launches += 2;
        }
        *launches += 1;
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    return cudaSuccess;
}

cudaError_t launch_dense_lu_c64(float2 *A, int32_t *piv, int32_t *info, float2 *dinv, int n, int N,
                                cudaStream_t s, int64_t *launches, unsigned int *status, bool tc) {
    return dense_lu_t<float2, NB_C64>(A, piv, info, dinv, n, N, s, launches, status, tc);
}
cudaError_t launch_dense_lu_c128(double2 *A, int32_t *piv, int32_t *info, double2 *dinv, int n, int N,
                                 cudaStream_t s, int64_t *launches) {
    return dense_lu_t<double2, NB_C128>(A, piv, info, dinv, n, N, s, launches, nullptr, false);
}

// chunks of LC right-hand sides: the widest (the factor is read once per chunk)
// of which there are still enough for the SMs, else the narrowest
static int ds_columns(int N, int L, int widest) {
    int dev = 0, sms = 152;
    if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    for (int lc = widest; lc > 4; lc /= 2)
        if ((int64_t)N * ((L + lc - 1) / lc) >= sms * 4 / 5) return lc;
    return 4;
}
constexpr int DS_GROUPED = 1024;  // largest order whose products are summed by eights
template <typename C, int NB, int LC, int TH>
static cudaError_t ds_launch(const C *A, const int32_t *piv, const C *dinv, C *B, int n, int N, int L,
                             const int32_t *skip, cudaStream_t s) {
    auto *kernel = n <= DS_GROUPED ? dense_solve_kernel<C, NB, LC, TH, false, 8>
                                   : dense_solve_kernel<C, NB, LC, TH, false, NB>;
    for (int p0 = 0; p0 < N; p0 += 65535) {  // grid.y limit
        const size_t nblk = ((size_t)n + NB - 1) / NB;
        kernel<<<dim3((L + LC - 1) / LC, std::min(N - p0, 65535)), TH, 0, s>>>(
            A + (size_t)p0 * n * n, piv + (size_t)p0 * n, dinv + p0 * nblk * 2 * NB * NB, B + (size_t)p0 * n * L, n, L,
            skip ? skip + p0 : nullptr);
    }
    return cudaGetLastError();
}
cudaError_t launch_dense_solve_c64(const float2 *A, const int32_t *piv, const float2 *dinv, float2 *B,
                                   int n, int N, int L, const int32_t *skip, cudaStream_t s) {
    switch (ds_columns(N, L, 16)) {
    case 16: return ds_launch<float2, NB_C64, 16, 512>(A, piv, dinv, B, n, N, L, skip, s);
    case 8: return ds_launch<float2, NB_C64, 8, 512>(A, piv, dinv, B, n, N, L, skip, s);
    default: return ds_launch<float2, NB_C64, 4, 512>(A, piv, dinv, B, n, N, L, skip, s);
    }
}
cudaError_t launch_dense_solve_c128(const double2 *A, const int32_t *piv, const double2 *dinv,
                                    double2 *B, int n, int N, int L, const int32_t *skip,
                                    cudaStream_t s) {
    if (ds_columns(N, L, 8) == 8) return ds_launch<double2, NB_C128, 8, 256>(A, piv, dinv, B, n, N, L, skip, s);
    return ds_launch<double2, NB_C128, 4, 256>(A, piv, dinv, B, n, N, L, skip, s);
}
// X = (P L U)^{-1}, n x n per point.  The composed interchanges take 2 n ints of
// shared memory; orders that have no room for them solve with the identity.
static constexpr int DINV_MAX = 4096;
__global__ void dense_identity_kernel(double2 *__restrict__ F, int n) {
    const int64_t nn = (int64_t)n * n;
    double2 *X = F + (size_t)blockIdx.y * nn;
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < nn; e += (int64_t)gridDim.x * blockDim.x)
        X[e] = make_double2(e % n == e / n ? 1.0 : 0.0, 0.0);
}
cudaError_t launch_dense_inverse_c128(const double2 *A, const int32_t *piv, const double2 *dinv, double2 *X, int n,
                                      int N, cudaStream_t s) {
    constexpr int LC = 8, TH = 256;
    const size_t nn = (size_t)n * n, nblk = ((size_t)n + NB_C128 - 1) / NB_C128;
    for (int p0 = 0; p0 < N; p0 += 65535) {  // grid.y limit
        const int np = std::min(N - p0, 65535);
        if (n > DINV_MAX) {
            dense_identity_kernel<<<dim3(grid_for_d((int64_t)nn, 256, 1024), np), 256, 0, s>>>(X + p0 * nn, n);
            const cudaError_t e = ds_launch<double2, NB_C128, LC, TH>(
                A + p0 * nn, piv + (size_t)p0 * n, dinv + p0 * nblk * 2 * NB_C128 * NB_C128, X + p0 * nn, n, np, n,
                nullptr, s);
            if (e != cudaSuccess) return e;
            continue;
        }
        dense_solve_kernel<double2, NB_C128, LC, TH, true, 8>
            <<<dim3((n + LC - 1) / LC, np), TH, sizeof(int) * (size_t)(2 * n), s>>>(
                A + p0 * nn, piv + (size_t)p0 * n, dinv + p0 * nblk * 2 * NB_C128 * NB_C128, X + p0 * nn, n, n,
                nullptr);
    }
    return cudaGetLastError();
}

cudaError_t launch_dense_residual(double2 *R, const double2 *T, const double2 *X, const double2 *U, int n, int L,
                                  int N, const int32_t *done, cudaStream_t s) {
    for (int p0 = 0; p0 < N; p0 += 65535) {  // grid.z limit
        const int np = std::min(N - p0, 65535);
        const size_t per = (size_t)n * L;
        dense_residual_kernel<<<dim3((n + DR_M - 1) / DR_M, (L + DR_N - 1) / DR_N, np), DR_THREADS, 0, s>>>(
            R + p0 * per, T + (size_t)p0 * n * n, X + p0 * per, U, done ? done + p0 : nullptr, n, L);
    }
    return cudaGetLastError();
}
cudaError_t launch_dense_colmax(const double2 *R, const double2 *X, int n, int L, int N, double *rmax,
                                double *xmax, const int32_t *done, cudaStream_t s) {
    for (int p0 = 0; p0 < N; p0 += 65535) {  // grid.y limit
        const size_t per = (size_t)n * L;
        dense_colmax_kernel<<<dim3(L, std::min(N - p0, 65535)), 256, 0, s>>>(
            R + p0 * per, X + p0 * per, n, L, rmax + (size_t)p0 * L, xmax + (size_t)p0 * L,
            done ? done + p0 : nullptr);
    }
    return cudaGetLastError();
}

cudaError_t launch_taylor_step(double2 *A, const double *pts, double2 c, double diag, int n, int p,
                               cudaStream_t s) {
    taylor_step_kernel<<<grid_for_d((int64_t)n * n, 256, 4096), 256, 0, s>>>(A, pts, c, diag, n, p);
    return cudaGetLastError();
}

cudaError_t launch_dense_eig_residual(const double2 *V, const double2 *lam, const double *pts,
                                      double diag, int n, int cnt, double *rr, double *vv, double *t1,
                                      cudaStream_t s) {
    dense_eig_residual_kernel<<<dim3((n + 127) / 128, cnt), 128, 0, s>>>(V, lam, pts, diag, n, rr, vv, t1);
    return cudaGetLastError();
}

}  // namespace rsrr
