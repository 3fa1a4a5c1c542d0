// FP64-accurate complex GEMM on the bf16 tensor cores by error-free slicing
// (the Ozaki scheme): C = alpha op(A) B + beta C with op(A) = A or A^H and
// real alpha, beta.  Used for the large products of the projection (Gram
// matrices of the sample block, Q^H R, R W, Q^H A_i Q) where native FP64
// runs at the GPU's reduced double-precision rate.
//
// 1. The complex product is one real product C~ = A~ B~ of depth K' = 2K
//    with Re/Im interleaved along K:
//      A~(i, 2k) = Re op(A)_ik,  A~(i, 2k+1) = Im op(A)_ik
//      B~(2k, j) = Re B_kj,  B~(2k+1, j) = -Im B_kj      (j < N:  Re C)
//      B~(2k, N+j) = Im B_kj,  B~(2k+1, N+j) = Re B_kj   (N + j: Im C)
// 2. Row i of A~ is scaled by 2^-e_i and column j of B~ by 2^-f_j with
//    2^(e-1) <= max |entry| < 2^e, then rounded to 55-bit fixed point
//    (exact for the largest entries, below 2^-55 absolute for the rest) and
//    split into 7 signed base-256 digits a_s in [-128, 128]:
//      x = sum_s a_s 2^(-7-8s).
//    Slice s is stored as the bf16 value a_s 2^(-8s) (exact).
// 3. Slice products of one group t = p + q are multiples of 2^(-8t) with an
//    integer part below 2^14 each; tensor-core FP32 sums of them stay exact
//    while the integer part is below 2^24.  Groups t = 0..4 get their own
//    accumulators and are folded into one int64 per output every 128 of K'
//    ((t+1) 128 2^14 <= 5 2^21 < 2^24): acc += 2^32 g_t.  Groups 5 and 6
//    (relative weight <= 2^-40) share one FP32 accumulator folded into an
//    FP32 sum; the tensor cores round such mixed-magnitude sums (measured:
//    a shared group-4..6 accumulator lost ~0.3 units of 2^-46), which at
//    this weight stays below 2^-54; the FP32 sum of at most 512 folds, each
//    below 2^-15.8 where a largest product is 2^14, rounds by less than 2^-54 K'
//    of that.  Pairs with t >= 7 (below 2^-56
//    relative) are dropped.  |acc| stays below K' 2^46 (every |x| < 1), so
//    K' <= 98304 keeps it below 2^62.6 (K is chunked beyond 49152).
// 4. C~_ij = 2^(e_i + f_j) 2^-46 (acc + 2^32 low), acc and the sum rounded to FP64.
#include <algorithm>
#include <climits>
#include <cmath>
#include <cstdint>
#include <cuda.h>
#include <cuda_bf16.h>
#include <mutex>
#include <string>

#include "rsrr.h"

#include "common.cuh"
#include "rsrr_internal.h"

namespace rsrr {

constexpr int OZ_S = 7;           // slices
constexpr int OZ_BM = 64;         // CTA tile rows (M)
constexpr int OZ_BN = 64;         // CTA tile columns (of the 2N real columns)
constexpr int OZ_KC = 32;         // K' per pipeline stage
constexpr int OZ_LD = OZ_KC + 8;  // shared-memory row length (bf16): 80 bytes, conflict-free ldmatrix
constexpr int OZ_NS = 3;          // pipeline stages
constexpr int OZ_FOLD = 4;        // stages per exact fold (K' = 128)
constexpr int OZ_BCACHE = 4;      // B slices held in registers per 16-deep step
constexpr int64_t OZ_KMAX = 49152;  // complex K per chunk: K' 2^46 < 2^63, the 64-bit sums do not overflow
constexpr int OZ_THREADS = 256;   // 8 warps: 2 (M) x 4 (N), 32 x 16 outputs each
constexpr int OZ_ROWS = OZ_S * (OZ_BM + OZ_BN);         // shared-memory rows per stage
constexpr int OZ_STAGE = OZ_ROWS * OZ_LD;                // bf16 elements per stage
constexpr size_t OZ_SMEM = sizeof(__nv_bfloat16) * OZ_STAGE * OZ_NS;  // 215040 bytes

// ----------------------------------------------------------- fixed point
// biased exponent field of |v|, subnormals and zero counted as 1
RSRR_DEV int exb_of(double v) {
    const int b = (int)((__double_as_longlong(v) >> 52) & 0x7FF);
    return b ? b : 1;
}

// round(v 2^(55 - e)) with e = E - 1022, E = largest biased exponent of the
// row; |result| <= 2^55.  Integer arithmetic only.
RSRR_DEV long long fixed55(double v, int E) {
    const long long bits = __double_as_longlong(v);
    int b = (int)((bits >> 52) & 0x7FF);
    long long mant = bits & 0xFFFFFFFFFFFFFll;
    if (b) mant |= 1ll << 52;
    else b = 1;
    const int sh = b - E + 2;  // <= 2
    long long m;
    if (sh >= 0) m = mant << sh;
    else if (sh > -62) m = (mant + (1ll << (-sh - 1))) >> (-sh);
    else m = 0;
    return bits < 0 ? -m : m;
}

// the 7 slices of a 55-bit fixed-point value as floats a_s 2^(-8s)
RSRR_DEV void digits7(long long m, float out[OZ_S]) {
#pragma unroll
    for (int s = 0; s < OZ_S - 1; ++s) {
        const int sh = 48 - 8 * s;
        const long long a = (m + (1ll << (sh - 1))) >> sh;  // round half up, |a| <= 128
        m -= a << sh;
        out[s] = (float)(int)a * ldexpf(1.f, -8 * s);
    }
    out[OZ_S - 1] = (float)(int)m * 0x1p-48f;  // remainder in [-128, 128)
}

// ----------------------------------------------------------- exponents
// E[c] = largest biased exponent in column c (contiguous, K entries); also
// written to E[c + dup] when dup > 0 (the Im-output columns of B~) and to E2[c]
__global__ void oz_colexp_kernel(int *__restrict__ E, const double2 *__restrict__ X, int64_t ld,
                                 int K, int cols, int dup, int *__restrict__ E2) {
    __shared__ int w[32];
    for (int c = blockIdx.x; c < cols; c += gridDim.x) {
        int m = 1;
        for (int k = threadIdx.x; k < K; k += blockDim.x) {
            const double2 v = X[(int64_t)c * ld + k];
            m = max(m, max(exb_of(v.x), exb_of(v.y)));
        }
        for (int off = 16; off; off >>= 1) m = max(m, __shfl_down_sync(0xffffffffu, m, off));
        if ((threadIdx.x & 31) == 0) w[threadIdx.x >> 5] = m;
        __syncthreads();
        if (threadIdx.x == 0) {
            int r = 1;
            for (int q = 0; q < (int)(blockDim.x >> 5); ++q) r = max(r, w[q]);
            E[c] = r;
            if (dup > 0) E[c + dup] = r;
            if (E2) E2[c] = r;
        }
        __syncthreads();
    }
}

// E[i] = max(E[i], largest biased exponent in row i of the column-major
// rows x K matrix X); E starts at 0.  Tiles of 32 rows x 256 columns.
__global__ void oz_rowexp_kernel(int *__restrict__ E, const double2 *__restrict__ X, int64_t ld,
                                 int rows, int K) {
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;  // 32 x 8
    const int i = blockIdx.x * 32 + tx;
    const int k0 = blockIdx.y * 256;
    int m = 1;
    if (i < rows)
        for (int k = k0 + ty; k < min(K, k0 + 256); k += 8) {
            const double2 v = X[(int64_t)k * ld + i];
            m = max(m, max(exb_of(v.x), exb_of(v.y)));
        }
    __shared__ int w[8][32];
    w[ty][tx] = m;
    __syncthreads();
    if (ty == 0 && i < rows) {
        for (int q = 1; q < 8; ++q) m = max(m, w[q][tx]);
        atomicMax(&E[i], m);
    }
}

// ----------------------------------------------------------- slicing
// Plane layout: P[s][r][k'], row length Kp (a multiple of 32), Rp rows.
RSRR_DEV void store_slices(__nv_bfloat16 *P, size_t stride, size_t off, double re, double im, int E) {
    float dr[OZ_S], di[OZ_S];
    digits7(fixed55(re, E), dr);
    digits7(fixed55(im, E), di);
#pragma unroll
    for (int s = 0; s < OZ_S; ++s)
        *reinterpret_cast<__nv_bfloat162 *>(P + s * stride + off) = __floats2bfloat162_rn(dr[s], di[s]);
}

RSRR_DEV void store_zero(__nv_bfloat16 *P, size_t stride, size_t off) {
    const __nv_bfloat162 z = __floats2bfloat162_rn(0.f, 0.f);
#pragma unroll
    for (int s = 0; s < OZ_S; ++s) *reinterpret_cast<__nv_bfloat162 *>(P + s * stride + off) = z;
}

// Rows built from contiguous columns of X.
//   mode 0 (A^H):  row r = conj(column r),                  r < R
//   mode 1 (B):    row r < H: (Re, -Im) of column r;  H <= r < 2H: (Im, Re) of column r - H
// Rows of columns >= R and k >= K are written as zeros.
__global__ void oz_slice_cols_kernel(__nv_bfloat16 *__restrict__ P, const int *__restrict__ E,
                                     const double2 *__restrict__ X, int64_t ld, int mode, int R,
                                     int H, int K, int Rp, int Kp) {
    const size_t stride = (size_t)Rp * Kp;
    const int Kh = Kp / 2;
    for (int r = blockIdx.y; r < Rp; r += gridDim.y) {
        const int c = (mode == 1 && r >= H) ? r - H : r;
        const int Ec = (c < R) ? E[c] : 1;
        for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < Kh; k += gridDim.x * blockDim.x) {
            const size_t off = (size_t)r * Kp + 2 * (size_t)k;
            if (c >= R || k >= K) {
                store_zero(P, stride, off);
                continue;
            }
            const double2 v = X[(int64_t)c * ld + k];
            double re = v.x, im = -v.y;
            if (mode == 1 && r >= H) { re = v.y; im = v.x; }
            store_slices(P, stride, off, re, im, Ec);
        }
    }
}

// Rows of A itself (column-major M x K, row i strided): 32 x 32 tiles
// transposed through shared memory.  Rows >= M and k >= K are zeros.
__global__ void oz_slice_rows_kernel(__nv_bfloat16 *__restrict__ P, const int *__restrict__ E,
                                     const double2 *__restrict__ A, int64_t lda, int M, int K, int Mp,
                                     int Kp) {
    __shared__ double2 t[32][33];
    const int i0 = blockIdx.x * 32, k0 = blockIdx.y * 32;
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;  // 32 x 8
    for (int r = ty; r < 32; r += 8) {
        const int i = i0 + tx, k = k0 + r;
        t[r][tx] = (i < M && k < K) ? A[(int64_t)k * lda + i] : make_double2(0.0, 0.0);
    }
    __syncthreads();
    const size_t stride = (size_t)Mp * Kp;
    const int Kh = Kp / 2;
    for (int r = ty; r < 32; r += 8) {
        const int i = i0 + r, k = k0 + tx;
        if (i >= Mp || k >= Kh) continue;
        const size_t off = (size_t)i * Kp + 2 * (size_t)k;
        if (i >= M || k >= K) {
            store_zero(P, stride, off);
            continue;
        }
        const double2 v = t[tx][r];
        store_slices(P, stride, off, v.x, v.y, E[i]);
    }
}

// Stage images for the tensor-core kernel: the slices of one operand tile
// (TR rows, 16 of K') stored in exactly the order that kernel keeps them in
// shared memory, so that one bulk copy moves one operand of a stage.
//   chunk (rb, ks): rows TR rb .. +TR-1, K' 16 ks .. +15; OZ_S TR 16 elements
//   element (s, row, k') of a chunk at  s ss + kc kcs + 8 (row % TR) + k' % 8,
//   kc = (k' % 16) / 8 the core-matrix column (8 rows x 16 bytes a core matrix)
//   per-slice operand (A):          ss = 16 TR,  kcs = 8 TR
//   slices stacked per core column (B, read as one N = 64 q operand):
//                                   ss = 8 TR,   kcs = 8 OZ_S TR
// One warp per 8 rows x 4 complex K (a core matrix of every slice): lane =
// 4 (row % 8) + k % 4, so every slice store of a warp is 128 contiguous bytes.
RSRR_DEV size_t tiled_offset(int r, int64_t kg, int lane, int64_t nks, int TR, bool stacked) {
    const size_t kcs = stacked ? 8 * (size_t)OZ_S * TR : 8 * (size_t)TR;
    const size_t chunk = (size_t)OZ_S * TR * 16;
    return ((size_t)(r / TR) * nks + (size_t)(kg >> 1)) * chunk + (size_t)(kg & 1) * kcs + 8 * (size_t)(r % TR) +
           2 * (lane & 3);
}
RSRR_DEV void store_digits(__nv_bfloat16 *P, size_t stride, size_t off, const float (&re)[OZ_S], const float (&im)[OZ_S]) {
#pragma unroll
    for (int s = 0; s < OZ_S; ++s)
        *reinterpret_cast<__nv_bfloat162 *>(P + s * stride + off) = __floats2bfloat162_rn(re[s], im[s]);
}

// The columns of X as rows: (Re, -Im) of column c to row c of PA (A^H, RA rows;
// may be null) and of PB, (Im, Re) to row H + c of PB (may be null).  Columns
// >= R and k >= K are zeros.  One pass serves both halves of B~ and, for a
// Hermitian product, A~ too: X is read and digitised once instead of three times.
__global__ void oz_slice_columns_kernel(__nv_bfloat16 *__restrict__ PA, int RA, __nv_bfloat16 *__restrict__ PB, int H,
                                        int Np, const int *__restrict__ E, const double2 *__restrict__ X, int64_t ld,
                                        int R, int K, int Kp, int TA, int TB) {
    const int lane = threadIdx.x & 31;
    const int rows = max(PA ? RA : 0, PB ? max(H, Np - 2 * H) : 0);
    const int64_t nkg = Kp / 8, total = (int64_t)((rows + 7) / 8) * nkg, nks = Kp / 16;
    const int64_t wstep = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t w = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; w < total; w += wstep) {
        const int64_t kg = w % nkg;  // consecutive warps along the columns
        const int c = (int)(8 * (w / nkg)) + (lane >> 2), k = (int)(4 * kg) + (lane & 3);
        float re[OZ_S], im[OZ_S], nim[OZ_S];
        double2 v = make_double2(0.0, 0.0);
        int e = 1;
        if (c < R && k < K) {
            v = X[(int64_t)c * ld + k];
            e = E[c];
        }
        digits7(fixed55(v.x, e), re);
        digits7(fixed55(-v.y, e), nim);
        if (PA && c < RA) store_digits(PA, 16 * (size_t)TA, tiled_offset(c, kg, lane, nks, TA, false), re, nim);
        if (PB && c < H) {
            digits7(fixed55(v.y, e), im);
            store_digits(PB, 8 * (size_t)TB, tiled_offset(c, kg, lane, nks, TB, true), re, nim);
            store_digits(PB, 8 * (size_t)TB, tiled_offset(H + c, kg, lane, nks, TB, true), im, re);
        }
        // rows of the last tile past the second half
        if (PB && c + 2 * H < Np) {
            const float z[OZ_S] = {};
            store_digits(PB, 8 * (size_t)TB, tiled_offset(c + 2 * H, kg, lane, nks, TB, true), z, z);
        }
    }
}

// Rows of the column-major X itself (A); rows >= R and k >= K are zeros.
__global__ void oz_slice_rows_tiled_kernel(__nv_bfloat16 *__restrict__ P, const int *__restrict__ E,
                                           const double2 *__restrict__ X, int64_t ld, int R, int K, int Rp, int Kp,
                                           int TR) {
    const int lane = threadIdx.x & 31;
    const int64_t nrg = Rp / 8, total = nrg * (Kp / 8), nks = Kp / 16;
    const int64_t wstep = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t w = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; w < total; w += wstep) {
        const int64_t rg = w % nrg, kg = w / nrg;  // consecutive warps along the rows
        const int r = (int)(8 * rg) + (lane >> 2), k = (int)(4 * kg) + (lane & 3);
        const size_t off = tiled_offset(r, kg, lane, nks, TR, false);
        if (r >= R || k >= K) {
            store_zero(P, 16 * (size_t)TR, off);
            continue;
        }
        const double2 v = X[(int64_t)k * ld + r];
        store_slices(P, 16 * (size_t)TR, off, v.x, v.y, E[r]);
    }
}

// ----------------------------------------------------------- the GEMM
RSRR_DEV void cp_async16(unsigned saddr, const void *gmem) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(saddr), "l"(gmem));
}
RSRR_DEV void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::); }
template <int N>
RSRR_DEV void cp_async_wait() { asm volatile("cp.async.wait_group %0;\n" ::"n"(N)); }

RSRR_DEV void ldmatrix_x4(unsigned r[4], unsigned saddr) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];\n"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(saddr));
}

RSRR_DEV void mma_bf16(float c[4], const unsigned a[4], unsigned b0, unsigned b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
        "{%0,%1,%2,%3};\n"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// round(f 2^32) for a group sum f of groups t <= 4, in integer instructions.
// Such an f is an integer multiple of 2^-32 below 2^24 in magnitude (step 3
// above), so f = m 2^(e-150) with a 24-bit m and e >= 95, and f 2^32 =
// m 2^(e-118) is an integer below 2^56: the shift loses only zero bits and
// the result is exactly the float-to-int64 conversion of f 2^32, without the
// conversion unit (it shares the GPU's slow double-precision pipe).
RSRR_DEV long long scaled_group_to_ll(float f) {
    const int bits = __float_as_int(f);
    const int e = (bits >> 23) & 0xFF;
    if (e == 0) return 0;  // +-0 (subnormals cannot occur: |f| >= 2^-32)
    long long m = (long long)((bits & 0x7FFFFF) | 0x800000);
    const int sh = e - 118;
    m = sh >= 0 ? (m << sh) : (m >> -sh);
    return bits < 0 ? -m : m;
}

// low (0 or at least 2^-48 in modulus) times 2^32 in FP64, by its bits
RSRR_DEV double low_value(float low) {
    const uint32_t b = (uint32_t)__float_as_int(low);
    const uint32_t e = (b >> 23) & 0xFF;
    if (e == 0 || e == 0xFF) return (double)low;  // zeros; infinities and NaN
    return __hiloint2double((int)((b & 0x80000000u) | (((b & 0x7FFFFFFFu) >> 3) + ((896u + 32u) << 20))), (int)(b << 29));
}

// 2^n (acc + 2^32 low), rounded once to FP64 in the sum.  The exponent is added and
// low converted in integers: the FP64 unit, whose instructions take 64 cycles a warp,
// is left with one conversion and one addition.
RSRR_DEV double oz_value(long long acc, float low, int n) {
    const double d = (double)acc + low_value(low);
    const long long b = __double_as_longlong(d);
    const int ex = (int)((b >> 52) & 0x7FF), nx = ex + n;
    if (ex >= 1 && ex <= 2046 && nx >= 1 && nx <= 2046) return __longlong_as_double(b + ((long long)n << 52));
    return ldexp(d, n);
}

// One CTA: a 64 x 64 tile of C~ over K' range [sp kchunk, (sp+1) kchunk).
// W != null: FP64 partial tile into W[sp][i][j'] (Mp x Np, row major).
// W == null: C = alpha C~ + beta C written directly (one split).
// upper_only: tiles strictly below the block diagonal of each half skip.
__global__ void __launch_bounds__(OZ_THREADS, 1)
oz_gemm_kernel(const __nv_bfloat16 *__restrict__ As, const __nv_bfloat16 *__restrict__ Bs,
               const int *__restrict__ Ea, const int *__restrict__ Eb, double *__restrict__ W,
               double2 *__restrict__ C, int64_t ldc, int M, int N, int H, int Mp, int Np, int Kp, int kchunk,
               int halfN_tiles, int upper_only, double alpha, double beta) {
    const int bm = blockIdx.x, bn = blockIdx.y, sp = blockIdx.z;
    if (upper_only && bm > (bn % halfN_tiles)) return;
    extern __shared__ __align__(128) unsigned char oz_smem[];
    const unsigned sbase = (unsigned)__cvta_generic_to_shared(oz_smem);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int wm = warp & 1, wn = warp >> 1;
    const int g = lane >> 2, tq = lane & 3;
    const int m0 = bm * OZ_BM, n0 = bn * OZ_BN;
    const int kbeg = sp * kchunk;
    const int kend = min(Kp, kbeg + kchunk);
    const int nk = kend > kbeg ? (kend - kbeg) / OZ_KC : 0;
    const size_t sA = (size_t)Mp * Kp, sB = (size_t)Np * Kp;

    float gs[6][2][2][4];
    long long acc[2][2][4];
    float low[2][2][4];
#pragma unroll
    for (int a = 0; a < 2; ++a)
#pragma unroll
        for (int b = 0; b < 2; ++b)
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                acc[a][b][q] = 0;
                low[a][b][q] = 0.f;
#pragma unroll
                for (int t = 0; t < 6; ++t) gs[t][a][b][q] = 0.f;
            }

    // stage rows: slice s, rows 0..63 from A~, 64..127 from B~
    auto load_stage = [&](int slot, int k0) {
        const unsigned dst = sbase + (unsigned)(slot * OZ_STAGE * 2);
        for (int q = tid; q < OZ_ROWS * 4; q += OZ_THREADS) {
            const int row = q >> 2, c = q & 3;
            const int s = row >> 7, rr = row & 127;
            const __nv_bfloat16 *src =
                (rr < OZ_BM) ? As + s * sA + (size_t)(m0 + rr) * Kp + k0 + c * 8
                             : Bs + s * sB + (size_t)(n0 + rr - OZ_BM) * Kp + k0 + c * 8;
            cp_async16(dst + (unsigned)((row * OZ_LD + c * 8) * 2), src);
        }
    };

#pragma unroll
    for (int st = 0; st < OZ_NS - 1; ++st) {
        if (st < nk) load_stage(st, kbeg + st * OZ_KC);
        cp_async_commit();
    }
    // per-lane ldmatrix row offsets (bf16 elements within one slice)
    const int li = lane & 7, mi = lane >> 3;
    const int a_off = (wm * 32 + (mi & 1) * 8 + li) * OZ_LD + (mi >> 1) * 8;
    const int b_off = (OZ_BM + wn * 16 + (mi >> 1) * 8 + li) * OZ_LD + (mi & 1) * 8;

    for (int it = 0; it < nk; ++it) {
        cp_async_wait<OZ_NS - 2>();
        __syncthreads();
        {
            const int nx = it + OZ_NS - 1;
            if (nx < nk) load_stage(nx % OZ_NS, kbeg + nx * OZ_KC);
            cp_async_commit();
        }
        const unsigned st = sbase + (unsigned)((it % OZ_NS) * OZ_STAGE * 2);
#pragma unroll
        for (int kk = 0; kk < OZ_KC; kk += 16) {
            // B slices 0..3 stay in registers for the whole step; 4..6 (used
            // by p <= 2 only) are loaded where needed
            unsigned bfr[OZ_BCACHE][4];
#pragma unroll
            for (int q = 0; q < OZ_BCACHE; ++q)
                ldmatrix_x4(bfr[q], st + (unsigned)((q * (OZ_BM + OZ_BN) * OZ_LD + b_off + kk) * 2));
#pragma unroll
            for (int p = 0; p < OZ_S; ++p) {
                unsigned afr[2][4];
                const unsigned pa = st + (unsigned)((p * (OZ_BM + OZ_BN) * OZ_LD + a_off + kk) * 2);
                ldmatrix_x4(afr[0], pa);
                ldmatrix_x4(afr[1], pa + 16 * OZ_LD * 2);
#pragma unroll
                for (int q = 0; q < OZ_S - p; ++q) {
                    const int t = p + q < 5 ? p + q : 5;
                    unsigned bx[4];
                    if (q < OZ_BCACHE) {
#pragma unroll
                        for (int r = 0; r < 4; ++r) bx[r] = bfr[q < OZ_BCACHE ? q : 0][r];
                    } else {
                        ldmatrix_x4(bx, st + (unsigned)((q * (OZ_BM + OZ_BN) * OZ_LD + b_off + kk) * 2));
                    }
#pragma unroll
                    for (int a = 0; a < 2; ++a)
#pragma unroll
                        for (int b = 0; b < 2; ++b) mma_bf16(gs[t][a][b], afr[a], bx[2 * b], bx[2 * b + 1]);
                }
            }
        }
        if ((it + 1) % OZ_FOLD == 0 || it == nk - 1) {
#pragma unroll
            for (int a = 0; a < 2; ++a)
#pragma unroll
                for (int b = 0; b < 2; ++b)
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
#pragma unroll
                        for (int t = 0; t < 5; ++t) {
                            acc[a][b][q] += scaled_group_to_ll(gs[t][a][b][q]);
                            gs[t][a][b][q] = 0.f;
                        }
                        low[a][b][q] += gs[5][a][b][q];
                        gs[5][a][b][q] = 0.f;
                    }
        }
    }
    cp_async_wait<0>();

#pragma unroll
    for (int a = 0; a < 2; ++a)
#pragma unroll
        for (int b = 0; b < 2; ++b)
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int i = m0 + wm * 32 + a * 16 + g + (q >= 2 ? 8 : 0);
                const int jj = n0 + wn * 16 + b * 8 + 2 * tq + (q & 1);
                const double v = oz_value(acc[a][b][q], low[a][b][q], Ea[i] + Eb[jj] - 2090);
                const int part = jj >= H, j = jj - part * H;
                if (W) {
                    W[(size_t)sp * Mp * Np + (size_t)i * Np + jj] = v;
                } else if (i < M && j < N) {
                    double *c = reinterpret_cast<double *>(C + (int64_t)j * ldc + i) + part;
                    double r = alpha * v;
                    if (beta != 0.0) r = fma(beta, *c, r);
                    *c = r;
                }
            }
}

// ----------------------------------------------------------- tcgen05 path
// The same products on the 5th-generation tensor cores: one CTA an SM takes 128 x
// 64 tiles of C~ in turn.  Per 16-deep stage of K' the 7 A slices (128
// rows) and the 7 B slices (64 rows each, stacked to 448 rows) arrive by two
// bulk copies of the TMA engine (the stage images of the slicing kernels,
// 28 and 14 KB, contiguous in global memory; issued by one thread, completion
// counted in bytes on the stage's mbarrier) in the K-major core-matrix layout
// (8 rows x 16 bytes per core matrix, no swizzle), in a ring of OZT_NST
// stages that runs on from tile to tile; a slot is refilled once the MMAs that read
// it have committed.  One thread issues
// 10 tcgen05.mma per stage (M = 128, N = 64..256, bf16 -> FP32 in tensor
// memory): every group t = p + q has its own 64-column region of tensor
// memory (7 regions, 448 of the 512 columns), so the pairs of one A slice
// (q = 0 .. 6 - p) are MMAs over consecutive B slices into consecutive
// regions, four slices (N = 256) at a time.  Groups t <= 4 hold at most
// (t+1) 2^14 per K' element, so every 192 of K' (and at the end of a tile) sixteen
// warps wait for the MMAs (tcgen05.commit -> mbarrier), read their part of the
// regions (tcgen05.ld; warp w of 16 reads TMEM lanes 32 (w % 4) .. +31 = tile
// rows, columns 16 (w / 4) .. +15), fold groups 0..4 into 64-bit integers and add
// groups 5..6 (relative weight <= 2^-40, rounded by design) into an FP32 sum;
// the next MMAs restart every region.  The copy and MMA threads are warps of their
// own, so while a tile's sums become FP64 results (12 000 cycles of the FP64 unit,
// as long as the MMAs of a 15-stage tile) the next tile's first MMAs run.
// Every mbarrier wait is bounded; a wait that runs out is
// counted in the caller's device status word and raises an abort flag in shared memory, upon
// which every role leaves its loop; the copies and MMAs already issued are waited for (bounded)
// before the CTA ends.
//
// What it measured: with one tile a CTA, folds and results behind CTA-wide barriers, a
// 30-stage tile took 100 000 cycles, 37 000 of them MMAs, 33 000 its results, 10 000
// folds, the rest waits for the ring to fill: 40000 x 237 x 237 899 us, 500 x 500 x 40000
// (Hermitian) 1534 us; now 534 and 1080 us.
constexpr int OZT_BM = 128;
constexpr int OZT_BN = 64;
constexpr int OZT_KC = 16;
constexpr int OZT_FOLDERS = 512;                 // 16 warps: 4 lane quarters x 4 column groups
constexpr int OZT_THREADS = OZT_FOLDERS + 64;    // and a warp each for the MMAs and the copies
constexpr int OZT_CPT = OZT_BN / (OZT_FOLDERS / 128);  // tile columns a thread folds (16)
constexpr int OZT_GM = 8;                        // row tiles of a group (order of the tiles)
constexpr int OZT_A_SLICE = OZT_BM * OZT_KC * 2;           // bytes of one A slice per stage
constexpr int OZT_B_SLICE = OZT_BN * OZT_KC * 2;           // bytes of one B slice per stage
constexpr int OZT_STAGE = OZ_S * (OZT_A_SLICE + OZT_B_SLICE);
constexpr int OZT_NST = 5;
// after the stages: 2 NST + 3 mbarriers, the TMEM address, the abort flag
constexpr int OZT_TSLOT = 16 * OZT_NST + 24;
constexpr int OZT_ABORT = OZT_TSLOT + 16;
constexpr size_t OZT_SMEM = (size_t)OZT_NST * OZT_STAGE + 128;
static_assert(OZT_ABORT + 4 <= 128, "barrier area");
static_assert(OZT_SMEM <= 232448, "shared memory per CTA");
// stage layout, K-major core matrices (8 rows x 16 bytes), no swizzle: per
// K-column of core matrices (8 of K) all rows of an operand are contiguous,
// 16 bytes a row, so one TMA box of 16 bytes x rows fills one such column
constexpr uint32_t OZT_SBO = 128;                          // next 8-row group
constexpr uint32_t OZT_LBO_A = OZT_BM * 16;                // next core column of an A slice
constexpr uint32_t OZT_LBO_B = OZ_S * OZT_BN * 16;         // next core column of the stacked B
constexpr int OZT_FOLD = 12;                      // stages per exact fold (K' = 192)
constexpr long long OZT_WAIT_LIMIT = 1LL << 22;
static_assert((4 + 1) * OZT_FOLD * OZT_KC * 16384 < (1 << 24), "group sums must stay exact in FP32");
static_assert(OZ_S * OZT_BN <= 512, "one tensor-memory region per group");

// shared-memory matrix descriptor: K-major, no swizzle, start / LBO (next core
// matrix along K) / SBO (next 8-row group) in 16-byte units, version 1
RSRR_DEV uint64_t umma_desc(uint32_t saddr, uint32_t lbo) {
    return (uint64_t)((saddr >> 4) & 0x3FFF) | ((uint64_t)((lbo >> 4) & 0x3FFF) << 16) |
           ((uint64_t)((OZT_SBO >> 4) & 0x3FFF) << 32) | (1ull << 46);
}
// instruction descriptor: bf16 x bf16 -> f32, both K-major, M = 128, N = n
RSRR_DEV uint32_t umma_idesc(int n) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(OZT_BM >> 4) << 24);
}
RSRR_DEV void umma_bf16(uint32_t d_tmem, uint64_t a, uint64_t b, uint32_t idesc, uint32_t accumulate) {
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
                 "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}\n"
                 ::"r"(d_tmem), "l"(a), "l"(b), "r"(idesc), "r"(accumulate) : "memory");
}
RSRR_DEV void umma_commit(uint32_t mbar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n"
                 ::"r"(mbar) : "memory");
}
// bulk copy (TMA engine) of `bytes` contiguous bytes into shared memory,
// completion counted in bytes on mbar; both addresses 16-byte aligned, bytes
// a multiple of 16
RSRR_DEV void bulk_load(uint32_t dst, const void *src, uint32_t bytes, uint32_t mbar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n"
                 ::"r"(dst), "l"(src), "r"(bytes), "r"(mbar) : "memory");
}
RSRR_DEV void mbar_expect_tx(uint32_t mbar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(mbar), "r"(bytes) : "memory");
}
RSRR_DEV bool mbar_wait(uint32_t mbar, uint32_t parity, long long limit = OZT_WAIT_LIMIT) {
    for (long long it = 0; it < limit; ++it) {
        uint32_t done;
        asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
                     "selp.u32 %0, 1, 0, p;\n\t}\n" : "=r"(done) : "r"(mbar), "r"(parity) : "memory");
        if (done) return true;
    }
    return false;
}
// bounded wait that also gives up as soon as another thread of the CTA has
// raised the abort flag, and raises it when it runs out (the final drain
// uses the plain bounded wait so that operations in flight still land)
RSRR_DEV bool mbar_wait_or_abort(uint32_t mbar, uint32_t parity, volatile int *abort_flag,
                                 long long limit = OZT_WAIT_LIMIT) {
    for (long long it = 0; it < limit; ++it) {
        uint32_t done;
        asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
                     "selp.u32 %0, 1, 0, p;\n\t}\n" : "=r"(done) : "r"(mbar), "r"(parity) : "memory");
        if (done) return true;
        if (*abort_flag) return false;
    }
    *abort_flag = 1;
    return false;
}
RSRR_DEV void tmem_ld16(uint32_t taddr, uint32_t (&r)[16]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];\n"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
}

// The integer n of a group sum g = n 2^(-8t) with |n| < 2^24 (t <= 4; the
// fold cadence bounds n), exactly, in FP32 and integer ALU operations (the
// conversion instructions are slow on this GPU).  s = 2^(8t), s12 = 2^(8t-12):
//   r  = fma(g, s12, 1.5 2^23) = 1.5 2^23 + h with h = rint(n 2^-12), |h| <= 2^12:
//        the sum lies in [2^23, 2^24), where floats are the integers
//   lo = n - 2^12 h (|lo| <= 2^11), an exact FMA;  r2 = 1.5 2^23 + lo, exact
//   bits(r) = 0x4B400000 + h and bits(r2) = 0x4B400000 + lo, so
//   n = 2^12 bits(r) + bits(r2) - 4097 0x4B400000  (mod 2^32; |n| < 2^31)
RSRR_DEV int group_int(float g, float s12, float s) {
    const float M = 12582912.f;  // 1.5 2^23
    const float r = fmaf(g, s12, M);
    const float lo = fmaf(r - M, -4096.f, g * s);
    const float r2 = lo + M;
    return (int)(((uint32_t)__float_as_int(r) << 12) + (uint32_t)__float_as_int(r2) - 4097u * 0x4B400000u);
}

// the work list: split sp, row tile bm, column tile bn of item w of `tiles` per split.
// Tiles go in groups of OZT_GM row tiles by all column tiles, row tiles first: the
// CTAs at work together share few stage images of either operand, which
// then come from L2.  Hermitian results: of each half the column tiles 2 bm ..
RSRR_DEV void ozt_item(int w, int tiles, int nbm, int nbn, int halfN_tiles, int upper_only, int &sp, int &bm, int &bn) {
    sp = w / tiles;
    int t = w % tiles;
    if (upper_only) {
        bm = 0;
        int cnt = halfN_tiles;  // column tiles of each half in row bm
        while (t >= 2 * cnt) {
            t -= 2 * cnt;
            ++bm;
            cnt -= OZT_BM / OZT_BN;
        }
        bn = (t / cnt) * halfN_tiles + (OZT_BM / OZT_BN) * bm + t % cnt;
    } else {
        const int grp = t / (OZT_GM * nbn), in = t % (OZT_GM * nbn);
        const int gm = min(OZT_GM, nbm - grp * OZT_GM);  // the last group may be narrower
        bm = grp * OZT_GM + in % gm;
        bn = in / gm;
    }
}

__global__ void __launch_bounds__(OZT_THREADS, 1)
oz_gemm_tc_kernel(const __nv_bfloat16 *__restrict__ As, const __nv_bfloat16 *__restrict__ Bs,
                  const int *__restrict__ Ea, const int *__restrict__ Eb, double *__restrict__ W,
                  double2 *__restrict__ C, int64_t ldc, int M, int N, int H, int Mp, int Np, int Kp, int kchunk,
                  int tiles, int items, int halfN_tiles, int upper_only, double alpha, double beta,
                  unsigned int *__restrict__ status) {
    extern __shared__ __align__(1024) unsigned char ozt_smem[];
    const uint32_t sbase = (uint32_t)__cvta_generic_to_shared(ozt_smem);
    const uint32_t mb_full = sbase + OZT_NST * OZT_STAGE;  // OZT_NST: stage's bytes landed (TMA)
    const uint32_t mb_empty = mb_full + 8 * OZT_NST;       // OZT_NST: stage's MMAs done
    const uint32_t mb_fold = mb_empty + 8 * OZT_NST;       // all MMAs so far done
    const uint32_t mb_free = mb_fold + 8;                  // regions read by the sixteen warps
    const uint32_t mb_done = mb_free + 8;                  // the MMAs still in flight at the end
    uint32_t *tslot = reinterpret_cast<uint32_t *>(ozt_smem + OZT_NST * OZT_STAGE + OZT_TSLOT);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(ozt_smem + OZT_NST * OZT_STAGE + OZT_ABORT);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int nbm = Mp / OZT_BM, nbn = Np / OZT_BN;
    auto stages = [&](int sp) {
        const int kbeg = sp * kchunk, kend = min(Kp, kbeg + kchunk);
        return kend > kbeg ? (kend - kbeg) / OZT_KC : 0;
    };

    if (tid == 0) {
        for (int q = 0; q < OZT_NST; ++q) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(mb_full + 8 * q));
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(mb_empty + 8 * q));
        }
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(mb_fold));
        asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(mb_free), "n"(OZT_FOLDERS / 32));
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(mb_done));
        *abort_flag = 0;
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;\n"
                     ::"r"((uint32_t)__cvta_generic_to_shared(tslot)));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n");
    }
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    const uint32_t tmem = *tslot;
    bool ok = true;

    if (warp == OZT_FOLDERS / 32) {  // ---- the MMAs
        if (lane == 0) {
            int slot = 0, folds = 0;
            uint32_t phase = 0;
            const uint64_t da = umma_desc(sbase, OZT_LBO_A), db = umma_desc(sbase + OZ_S * OZT_A_SLICE, OZT_LBO_B);
            for (int w = blockIdx.x; ok && w < items; w += gridDim.x) {
                int sp, bm, bn;
                ozt_item(w, tiles, nbm, nbn, halfN_tiles, upper_only, sp, bm, bn);
                const int nk = stages(sp);
                for (int it = 0, left = 0; it < nk; ++it) {
                    const uint32_t keep = left != 0;  // all regions restart after a fold
                    if (left == 0) {
                        left = min(OZT_FOLD, nk - it);
                        if (folds > 0 && !mbar_wait_or_abort(mb_free, (folds - 1) & 1, abort_flag)) { ok = false; break; }
                    }
                    if (!mbar_wait_or_abort(mb_full + 8 * slot, phase, abort_flag)) { ok = false; break; }
                    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
                    const uint64_t so = (uint64_t)((slot * OZT_STAGE) >> 4);
#pragma unroll
                    for (int p = 0; p < OZ_S; ++p) {
                        // groups p .. 6 (q = 0 .. 6 - p): consecutive B slices into
                        // consecutive regions, at most 4 slices (N = 256) per MMA
#pragma unroll
                        for (int q0 = 0; q0 <= OZ_S - 1 - p; q0 += 4) {
                            const int nq = min(4, OZ_S - p - q0);
                            umma_bf16(tmem + (uint32_t)((p + q0) * OZT_BN), da + so + ((p * OZT_A_SLICE) >> 4),
                                      db + so + ((q0 * OZT_BN * 16) >> 4), umma_idesc(nq * OZT_BN), p == 0 ? keep : 1u);
                        }
                    }
                    umma_commit(mb_empty + 8 * slot);
                    if (--left == 0) {
                        umma_commit(mb_fold);
                        ++folds;
                    }
                    if (++slot == OZT_NST) {
                        slot = 0;
                        phase ^= 1;
                    }
                }
            }
            umma_commit(mb_done);
            ok = mbar_wait(mb_done, 0) && ok;
        }
        __syncwarp();
    } else if (warp == OZT_FOLDERS / 32 + 1) {  // ---- the copies
        if (lane == 0) {
            const size_t nks = (size_t)(Kp / OZT_KC);
            int issued = 0;  // stages whose copies were issued (all of them unless a wait ran out)
            for (int w = blockIdx.x; ok && w < items; w += gridDim.x) {
                int sp, bm, bn;
                ozt_item(w, tiles, nbm, nbn, halfN_tiles, upper_only, sp, bm, bn);
                const int nk = stages(sp);
                const size_t k0 = (size_t)(sp * kchunk / OZT_KC);
                const __nv_bfloat16 *srcA = As + ((size_t)bm * nks + k0) * (OZ_S * OZT_BM * OZT_KC);
                const __nv_bfloat16 *srcB = Bs + ((size_t)bn * nks + k0) * (OZ_S * OZT_BN * OZT_KC);
                for (int st = 0; st < nk; ++st) {
                    const int slot = issued % OZT_NST;
                    // the slot was last read by the MMAs of stage issued - NST
                    if (issued >= OZT_NST &&
                        !mbar_wait_or_abort(mb_empty + 8 * slot, ((issued / OZT_NST) - 1) & 1, abort_flag)) {
                        ok = false;
                        break;
                    }
                    const uint32_t full = mb_full + 8 * slot;
                    mbar_expect_tx(full, (uint32_t)OZT_STAGE);
                    const uint32_t a0 = sbase + (uint32_t)(slot * OZT_STAGE);
                    const uint32_t b0 = a0 + OZ_S * OZT_A_SLICE;
                    bulk_load(a0, srcA + (size_t)st * (OZ_S * OZT_BM * OZT_KC), (uint32_t)(OZ_S * OZT_A_SLICE), full);
                    bulk_load(b0, srcB + (size_t)st * (OZ_S * OZT_BN * OZT_KC), (uint32_t)(OZ_S * OZT_B_SLICE), full);
                    ++issued;
                }
            }
            // every copy that was issued has landed before the CTA leaves (waits
            // bounded; the last issued stage of each slot is its latest phase)
            for (int st = max(0, issued - OZT_NST); st < issued; ++st)
                ok = mbar_wait(mb_full + 8 * (st % OZT_NST), (st / OZT_NST) & 1) && ok;
        }
        __syncwarp();
    } else {  // ---- folds and results
        const int lrow = 32 * (warp & 3) + lane, lcol = OZT_CPT * (warp >> 2);
        const uint32_t tpart = tmem + ((uint32_t)(32 * (warp & 3)) << 16) + (uint32_t)lcol;
        int folds = 0;
        for (int w = blockIdx.x; w < items; w += gridDim.x) {
            int sp, bm, bn;
            ozt_item(w, tiles, nbm, nbn, halfN_tiles, upper_only, sp, bm, bn);
            long long acc[OZT_CPT];
            float low[OZT_CPT];
#pragma unroll
            for (int c = 0; c < OZT_CPT; ++c) {
                acc[c] = 0;
                low[c] = 0.f;
            }
            for (int nk = stages(sp); nk > 0; nk -= OZT_FOLD) {
                ok = __all_sync(0xffffffffu, mbar_wait_or_abort(mb_fold, folds & 1, abort_flag));
                if (!ok) break;
                ++folds;
                asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
                static_assert(OZT_CPT == 16, "one 16-column TMEM load per region");
#pragma unroll
                for (int t = 0; t < OZ_S; ++t) {
                    uint32_t r[16];
                    tmem_ld16(tpart + (uint32_t)(t * OZT_BN), r);
                    if (t == OZ_S - 1) {  // regions free again
                        asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
                        if (lane == 0)
                            asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(mb_free) : "memory");
                    }
#pragma unroll
                    for (int j = 0; j < 16; ++j) {
                        if (t < 5)
                            acc[j] += (long long)group_int(__uint_as_float(r[j]), 0x1p-12f * (float)(1ull << (8 * t)),
                                                           (float)(1ull << (8 * t)))
                                      << (32 - 8 * t);
                        else
                            low[j] += __uint_as_float(r[j]);
                    }
                }
            }
            if (!ok) break;
            const int i = bm * OZT_BM + lrow, j0 = bn * OZT_BN + lcol;
            const int ea = Ea[i] - 2090;
            if (W) {
                double2 *wp = reinterpret_cast<double2 *>(W + (size_t)sp * Mp * Np + (size_t)i * Np + j0);
#pragma unroll
                for (int c = 0; c < OZT_CPT; c += 2)
                    wp[c / 2] = make_double2(oz_value(acc[c], low[c], ea + Eb[j0 + c]),
                                             oz_value(acc[c + 1], low[c + 1], ea + Eb[j0 + c + 1]));
                continue;
            }
            if (i >= M) continue;
#pragma unroll
            for (int c0 = 0; c0 < OZT_CPT; c0 += 8) {  // the reads of C ahead of its writes
                double old[8];
                double *cp[8];
#pragma unroll
                for (int c = 0; c < 8; ++c) {
                    const int jj = j0 + c0 + c, part = jj >= H, j = jj - part * H;
                    cp[c] = j < N ? reinterpret_cast<double *>(C + (int64_t)j * ldc + i) + part : nullptr;
                    old[c] = cp[c] && beta != 0.0 ? *cp[c] : 0.0;
                }
#pragma unroll
                for (int c = 0; c < 8; ++c) {
                    const double v = oz_value(acc[c0 + c], low[c0 + c], ea + Eb[j0 + c0 + c]);
                    double r = alpha == 1.0 ? v : alpha * v;
                    if (beta != 0.0) r = fma(beta, old[c], r);
                    if (cp[c]) *cp[c] = r;
                }
            }
        }
    }
    if (!ok && lane == 0) atomicAdd(status, 1u);
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;\n" ::"r"(tmem));
}

// Failure-detection check of the bounded wait: one thread waits on an
// mbarrier that nothing arrives on; the wait gives up after `limit` tries and
// is counted in the status word, exactly as in the tensor-core kernel.
__global__ void ozt_wait_check_kernel(long long limit, unsigned int *status) {
    __shared__ __align__(8) unsigned long long bar;
    if (threadIdx.x != 0) return;
    const uint32_t a = (uint32_t)__cvta_generic_to_shared(&bar);
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(a) : "memory");
    if (!mbar_wait(a, 0, limit)) atomicAdd(status, 1u);
}

cudaError_t launch_wait_check(long long limit, unsigned int *status, cudaStream_t s) {
    ozt_wait_check_kernel<<<1, 32, 0, s>>>(limit, status);
    return cudaGetLastError();
}

// C = alpha sum_s W[s] + beta C (fixed order over the splits: four sums of every
// fourth one, whose roundings are of a quarter of the whole: 32 splits of one-sign
// data, 24 x 24 of depth 33000, rms error 1.4e-16 in one chain, 5.9e-17 so)
__global__ void oz_combine_kernel(double2 *__restrict__ C, int64_t ldc, const double *__restrict__ W,
                                  int M, int N, int H, int Mp, int Np, int splits, double alpha, double beta,
                                  int upper_only, int bm) {
    const int64_t total = (int64_t)M * N;
    for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < total;
         q += (int64_t)gridDim.x * blockDim.x) {
        const int i = (int)(q % M), j = (int)(q / M);
        if (upper_only && bm * (i / bm) > OZ_BN * (j / OZ_BN) + OZ_BN - 1) continue;
        double re[4] = {}, im[4] = {};
        for (int s = 0; s < splits; s += 4)
#pragma unroll
            for (int u = 0; u < 4; ++u)
                if (s + u < splits) {
                    const double *Wp = W + (size_t)(s + u) * Mp * Np + (size_t)i * Np;
                    re[u] += Wp[j];
                    im[u] += Wp[H + j];
                }
        double2 r = make_double2(alpha * ((re[0] + re[1]) + (re[2] + re[3])), alpha * ((im[0] + im[1]) + (im[2] + im[3])));
        if (beta != 0.0) {
            const double2 c = C[(int64_t)j * ldc + i];
            r.x = fma(beta, c.x, r.x);
            r.y = fma(beta, c.y, r.y);
        }
        C[(int64_t)j * ldc + i] = r;
    }
}

__global__ void oz_mirror_kernel(double2 *__restrict__ C, int64_t ldc, int n) {
    const int64_t total = (int64_t)n * n;
    for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < total;
         q += (int64_t)gridDim.x * blockDim.x) {
        const int i = (int)(q % n), j = (int)(q / n);
        if (i > j) {
            const double2 v = C[(int64_t)i * ldc + j];
            C[(int64_t)j * ldc + i] = make_double2(v.x, -v.y);
        } else if (i == j) {
            C[(int64_t)j * ldc + i].y = 0.0;  // the rounded low groups leave ~2^-56 here
        }
    }
}

// C = beta C (K = 0 or alpha = 0)
__global__ void oz_scale_kernel(double2 *__restrict__ C, int64_t ldc, int M, int N, double beta) {
    const int64_t total = (int64_t)M * N;
    for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < total;
         q += (int64_t)gridDim.x * blockDim.x) {
        const int i = (int)(q % M), j = (int)(q / M);
        double2 &c = C[(int64_t)j * ldc + i];
        c = beta == 0.0 ? make_double2(0.0, 0.0) : make_double2(beta * c.x, beta * c.y);
    }
}

// ----------------------------------------------------------- host side
static int64_t rup(int64_t x, int64_t m) { return (x + m - 1) / m * m; }
static int grid_for(int64_t work) {
    return (int)std::max<int64_t>(1, std::min<int64_t>((work + 255) / 256, 152 * 8));
}

namespace {
struct OzPlan {
    int64_t Mp, Np, Kc, Kp;  // Kc: complex K per chunk
    int64_t H;               // first column of C~ that holds imaginary parts
    int splits;
    int64_t kchunk;          // K' per split
    size_t bytes;
};

size_t plan_bytes(int64_t Mp, int64_t Np, int64_t Kp, int splits) {
    size_t b = rup((int64_t)sizeof(__nv_bfloat16) * OZ_S * Mp * Kp, 256);
    b += rup((int64_t)sizeof(__nv_bfloat16) * OZ_S * Np * Kp, 256);
    b += rup((int64_t)sizeof(int) * (Mp + Np), 256);
    if (splits > 1) b += rup((int64_t)sizeof(double) * splits * Mp * Np, 256);
    return b;
}

// splits of K that balance the waves over the 152 SMs (one CTA per SM)
int choose_splits(int64_t tiles, int64_t Kp) {
    int best = 1;
    double best_cost = 1e300;
    for (int s = 1; s <= 32; ++s) {
        if (s > 1 && Kp / s < (int64_t)OZ_FOLD * OZ_KC * 2) break;
        const double waves = (double)((tiles * s + 151) / 152);
        const double cost = waves / s * (1.0 + 0.01 * s);
        if (cost < best_cost - 1e-12) {
            best_cost = cost;
            best = s;
        }
    }
    return best;
}

// computed tiles of a bm x 64 tiling (upper block triangle only for Hermitian results)
int64_t tile_count(int64_t Mp, int64_t Np, int bm, bool upper, int64_t halfN) {
    if (!upper) return (Mp / bm) * (Np / OZ_BN);
    int64_t t = 0;
    for (int64_t a = 0; a < Mp / bm; ++a)
        for (int64_t b = 0; b < Np / OZ_BN; ++b)
            if (bm * a <= OZ_BN * (b % halfN) + OZ_BN - 1) ++t;
    return t;
}

OzPlan make_plan(int M, int N, int K, bool hermitian, size_t ws_bytes, int bm, int64_t kmax = OZ_KMAX,
                 bool packed = false) {
    OzPlan p{};
    p.Mp = rup(M, bm);
    // a Hermitian result's halves start on tiles of their own, so that the tiles
    // below the diagonal of both can be left out (packed: they do not, for
    // ozaki_padding_bytes)
    p.H = hermitian && !packed ? rup(N, OZ_BN) : N;
    p.Np = rup(2 * p.H, OZ_BN);
    const int64_t tiles = packed ? (p.Mp / bm) * (p.Np / OZ_BN) / 2
                                 : tile_count(p.Mp, p.Np, bm, hermitian, hermitian ? p.H / OZ_BN : p.Np / OZ_BN);
    const int64_t Kall = std::max(K, 1);
    auto fit = [&](int64_t kc) {
        p.Kc = kc;
        p.Kp = rup(2 * p.Kc, OZ_KC);
        p.splits = choose_splits(std::max<int64_t>(tiles, 1), p.Kp);
        while (p.splits > 1 && plan_bytes(p.Mp, p.Np, p.Kp, p.splits) > ws_bytes) --p.splits;
        p.bytes = plan_bytes(p.Mp, p.Np, p.Kp, p.splits);
        return p.bytes <= ws_bytes;
    };
    // the fewest chunks of equal depth that fit
    int64_t nch = (Kall + kmax - 1) / kmax;
    while (!fit(rup((Kall + nch - 1) / nch, 16)) && p.Kc > 16) nch *= 2;
    p.kchunk = rup((p.Kp + p.splits - 1) / p.splits, OZ_KC);
    p.splits = (int)((p.Kp + p.kchunk - 1) / p.kchunk);
    return p;
}
}  // namespace

static size_t planned_bytes(int M, int N, int K, bool hermitian, int64_t kmax, bool packed) {
    if (kmax <= 0 || kmax > OZ_KMAX) kmax = OZ_KMAX;
    return std::max(make_plan(M, N, K, hermitian, SIZE_MAX, OZ_BM, kmax, packed).bytes,
                    make_plan(M, N, K, hermitian, SIZE_MAX, OZT_BM, kmax, packed).bytes);
}
size_t ozaki_workspace_bytes(int M, int N, int K, bool hermitian, int64_t kmax) {
    return planned_bytes(M, N, K, hermitian, kmax, false);
}
size_t ozaki_padding_bytes(int N, int K, int64_t kmax) {
    const size_t padded = planned_bytes(N, N, K, true, kmax, false), packed = planned_bytes(N, N, K, true, kmax, true);
    return padded > packed ? padded - packed : 0;
}

double ozaki_tc_flops(int M, int N, int K, bool hermitian, bool legacy) {
    if (M <= 0 || N <= 0 || K <= 0) return 0.0;
    const int bm = legacy ? OZ_BM : OZT_BM;
    const bool upper = hermitian && M == N;
    const OzPlan p = make_plan(M, N, K, upper, SIZE_MAX, bm);
    const double pairs = OZ_S * (OZ_S + 1) / 2;
    const double tiles = (double)tile_count(p.Mp, p.Np, bm, upper, upper ? p.H / OZ_BN : p.Np / OZ_BN);
    return 2.0 * pairs * tiles * bm * OZ_BN * (double)p.Kp;
}

cudaError_t ozaki_zgemm(int M, int N, int K, bool conjA, const double2 *A, int64_t lda,
                        const double2 *B, int64_t ldb, double2 *C, int64_t ldc, double alpha,
                        double beta, bool hermitian, void *ws, size_t ws_bytes, cudaStream_t s,
                        int64_t *launches, EventPool *timer, double *tc_flops, bool legacy,
                        unsigned int *status) {
    if (M <= 0 || N <= 0) return cudaSuccess;
    if (!legacy && !status) return cudaErrorInvalidValue;
    cudaError_t e;
    if (K <= 0 || alpha == 0.0) {
        oz_scale_kernel<<<grid_for((int64_t)M * N), 256, 0, s>>>(C, ldc, M, N, beta);
        if (launches) *launches += 1;
        return cudaGetLastError();
    }
    if (hermitian && (M != N || !conjA || A != B || lda != ldb)) hermitian = false;
    const int bm = legacy ? OZ_BM : OZT_BM;
    const OzPlan p = make_plan(M, N, K, hermitian, ws_bytes, bm);
    if (p.bytes > ws_bytes) return cudaErrorMemoryAllocation;
    if (legacy)
        e = cudaFuncSetAttribute(oz_gemm_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)OZ_SMEM);
    else
        e = cudaFuncSetAttribute(oz_gemm_tc_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)OZT_SMEM);
    int dev = 0, nsm = 152;
    if (e == cudaSuccess) e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    char *w = static_cast<char *>(ws);
    __nv_bfloat16 *As = reinterpret_cast<__nv_bfloat16 *>(w);
    w += rup((int64_t)sizeof(__nv_bfloat16) * OZ_S * p.Mp * p.Kp, 256);
    __nv_bfloat16 *Bs = reinterpret_cast<__nv_bfloat16 *>(w);
    w += rup((int64_t)sizeof(__nv_bfloat16) * OZ_S * p.Np * p.Kp, 256);
    int *Ea = reinterpret_cast<int *>(w);
    int *Eb = Ea + p.Mp;
    w += rup((int64_t)sizeof(int) * (p.Mp + p.Np), 256);
    double *Wp = p.splits > 1 ? reinterpret_cast<double *>(w) : nullptr;
    const bool upper = hermitian;
    const int H = (int)p.H, halfN_tiles = (int)(upper ? p.H / OZ_BN : p.Np / OZ_BN);

    for (int64_t kc0 = 0; kc0 < K; kc0 += p.Kc) {
        const int Kc = (int)std::min<int64_t>(p.Kc, K - kc0);
        const double b = kc0 == 0 ? beta : 1.0;
        const double2 *Ak = conjA ? A + kc0 : A + kc0 * lda;
        const double2 *Bk = B + kc0;
        if ((e = cudaMemsetAsync(Ea, 0, sizeof(int) * (p.Mp + p.Np), s)) != cudaSuccess) return e;
        if (conjA && !hermitian)
            oz_colexp_kernel<<<std::min(M, 65535), 256, 0, s>>>(Ea, Ak, lda, Kc, M, 0, nullptr);
        else if (!conjA)
            oz_rowexp_kernel<<<dim3((unsigned)((M + 31) / 32), (unsigned)((Kc + 255) / 256)), 256, 0, s>>>(
                Ea, Ak, lda, M, Kc);
        oz_colexp_kernel<<<std::min(N, 65535), 256, 0, s>>>(Eb, Bk, ldb, Kc, N, H, hermitian ? Ea : nullptr);
        if (legacy) {
            const int kx = (int)std::min<int64_t>((p.Kp / 2 + 255) / 256, 64);
            if (conjA)
                oz_slice_cols_kernel<<<dim3(kx, (unsigned)std::min<int64_t>(p.Mp, 65535)), 256, 0, s>>>(
                    As, Ea, Ak, lda, 0, M, M, Kc, (int)p.Mp, (int)p.Kp);
            else
                oz_slice_rows_kernel<<<dim3((unsigned)(p.Mp / 32), (unsigned)((p.Kp / 2 + 31) / 32)), 256, 0,
                                       s>>>(As, Ea, Ak, lda, M, Kc, (int)p.Mp, (int)p.Kp);
            oz_slice_cols_kernel<<<dim3(kx, (unsigned)std::min<int64_t>(p.Np, 65535)), 256, 0, s>>>(
                Bs, Eb, Bk, ldb, 1, N, H, Kc, (int)p.Np, (int)p.Kp);
        } else {
            // stage images: one warp per 8 rows x 8 of K'
            auto blocks = [](int64_t rows, int64_t kp) {
                return (unsigned)std::max<int64_t>(1, std::min<int64_t>(rows / 8 * (kp / 8) / 8, 152 * 16));
            };
            if (!hermitian) {
                if (conjA)
                    oz_slice_columns_kernel<<<blocks(p.Mp, p.Kp), 256, 0, s>>>(As, (int)p.Mp, nullptr, 0, 0, Ea, Ak, lda,
                                                                               M, Kc, (int)p.Kp, OZT_BM, OZT_BN);
                else
                    oz_slice_rows_tiled_kernel<<<blocks(p.Mp, p.Kp), 256, 0, s>>>(As, Ea, Ak, lda, M, Kc, (int)p.Mp,
                                                                                  (int)p.Kp, OZT_BM);
            }
            oz_slice_columns_kernel<<<blocks(std::max(p.Mp, p.H), p.Kp), 256, 0, s>>>(
                hermitian ? As : nullptr, (int)p.Mp, Bs, H, (int)p.Np, Eb, Bk, ldb, N, Kc, (int)p.Kp, OZT_BM, OZT_BN);
        }
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
        const unsigned tm = (unsigned)(p.Mp / bm), tn = (unsigned)(p.Np / OZ_BN);
        const int64_t tiles = tile_count(p.Mp, p.Np, bm, upper, halfN_tiles), items = tiles * p.splits;
        if (!legacy && items > INT_MAX) return cudaErrorInvalidValue;
        const dim3 grid = legacy ? dim3(tm, tn, (unsigned)p.splits) : dim3((unsigned)std::min<int64_t>(items, nsm));
        cudaEvent_t ev1 = nullptr;
        if (timer) {
            cudaEvent_t ev0;
            if ((e = timer->next(&ev0)) != cudaSuccess) return e;
            if ((e = timer->next(&ev1)) != cudaSuccess) return e;
            if ((e = cudaEventRecord(ev0, s)) != cudaSuccess) return e;
        }
        if (legacy)
            oz_gemm_kernel<<<grid, OZ_THREADS, OZ_SMEM, s>>>(As, Bs, Ea, Eb, Wp, C, ldc, M, N, H, (int)p.Mp,
                                                            (int)p.Np, (int)p.Kp, (int)p.kchunk,
                                                            halfN_tiles, upper ? 1 : 0, alpha, b);
        else
            oz_gemm_tc_kernel<<<grid, OZT_THREADS, OZT_SMEM, s>>>(As, Bs, Ea, Eb, Wp, C, ldc, M, N, H,
                                                                 (int)p.Mp, (int)p.Np, (int)p.Kp,
                                                                 (int)p.kchunk, (int)tiles, (int)items, halfN_tiles,
                                                                 upper ? 1 : 0, alpha, b, status);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
        if (timer && (e = cudaEventRecord(ev1, s)) != cudaSuccess) return e;
        if (tc_flops) *tc_flops += ozaki_tc_flops(M, N, Kc, upper, legacy);
        if (Wp) {
            oz_combine_kernel<<<grid_for((int64_t)M * N), 256, 0, s>>>(C, ldc, Wp, M, N, H, (int)p.Mp,
                                                                       (int)p.Np, p.splits, alpha, b,
                                                                       upper ? 1 : 0, bm);
            if ((e = cudaGetLastError()) != cudaSuccess) return e;
        }
        if (launches) *launches += (hermitian && !legacy ? 3 : 5) + (Wp ? 1 : 0);
    }
    if (hermitian) {  // exactly Hermitian result, whether or not tiles were skipped
        oz_mirror_kernel<<<grid_for((int64_t)M * M), 256, 0, s>>>(C, ldc, M);
        if (launches) *launches += 1;
    }
    return cudaGetLastError();
}

}  // namespace rsrr

// ----------------------------------------------------------- C ABI
namespace rsrr {
std::string &thread_error();  // api.cu: last error of a handle-less call

// Work space of rsrr_zgemm: a stream-ordered pool per device that keeps at most
// ZGEMM_KEEP bytes between calls (mapping and unmapping 1.7 GB took 1.15 ms of a
// 40000 x 500 Gram matrix's 3.4); allocations and frees are ordered on the
// caller's stream, so threads and streams do not share a block in use.  What is
// kept is given back when a handle or a server is created, and when an
// allocation of the pool fails; the driver takes it back by itself for any other
// allocation that does not fit beside it.  A pool is not among what a
// cudaDeviceReset destroys: it serves the next context as before.
constexpr uint64_t ZGEMM_KEEP = 2ull << 30;
constexpr int ZGEMM_DEVICES = 64;
static std::mutex g_zgemm_mu;
static cudaMemPool_t g_zgemm_pool[ZGEMM_DEVICES] = {};

static cudaMemPool_t zgemm_pool() {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= ZGEMM_DEVICES) return nullptr;
    std::lock_guard<std::mutex> lk(g_zgemm_mu);
    if (!g_zgemm_pool[dev]) {
        cudaMemPoolProps props = {};
        props.allocType = cudaMemAllocationTypePinned;
        props.location.type = cudaMemLocationTypeDevice;
        props.location.id = dev;
        cudaMemPool_t pool = nullptr;
        if (cudaMemPoolCreate(&pool, &props) != cudaSuccess) {
            cudaGetLastError();
            return nullptr;
        }
        uint64_t keep = ZGEMM_KEEP;
        if (cudaMemPoolSetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &keep) != cudaSuccess) {
            cudaGetLastError();
            cudaMemPoolDestroy(pool);
            return nullptr;
        }
        g_zgemm_pool[dev] = pool;
    }
    return g_zgemm_pool[dev];
}

void zgemm_release_kept() {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= ZGEMM_DEVICES) {
        cudaGetLastError();
        return;
    }
    std::lock_guard<std::mutex> lk(g_zgemm_mu);
    if (g_zgemm_pool[dev] && cudaMemPoolTrimTo(g_zgemm_pool[dev], 0) != cudaSuccess) cudaGetLastError();
}

namespace {
// one call's work space; freed on the stream it was allocated on
struct ZgemmWs {
    void *p = nullptr;
    bool pooled = false;
    cudaStream_t s;
    explicit ZgemmWs(cudaStream_t stream) : s(stream) {}
    cudaError_t get(size_t bytes) {
        cudaError_t e = cudaErrorMemoryAllocation;
        if (cudaMemPool_t pool = zgemm_pool()) {
            e = cudaMallocFromPoolAsync(&p, bytes, pool, s);
            pooled = e == cudaSuccess;
            if (!pooled) cudaGetLastError();
        }
        if (!pooled) {
            zgemm_release_kept();
            e = cudaMalloc(&p, bytes);
        }
        return e;
    }
    ~ZgemmWs() {
        if (p && pooled) cudaFreeAsync(p, s);
        else if (p) cudaFree(p);
    }
};
}  // namespace
}  // namespace rsrr

extern "C" rsrr_status rsrr_zgemm(int32_t M, int32_t N, int32_t K, int32_t conjA, const rsrr_c128 *A,
                                  int64_t lda, const rsrr_c128 *B, int64_t ldb, rsrr_c128 *C,
                                  int64_t ldc, double alpha, double beta, int32_t method,
                                  int32_t hermitian, size_t max_ws_bytes, void *stream) {
    using namespace rsrr;
    auto fail = [](rsrr_status st, const char *what, cudaError_t e = cudaSuccess) {
        std::string m = std::string("rsrr_zgemm: ") + what;
        if (e != cudaSuccess) m += std::string(": ") + cudaGetErrorString(e);
        thread_error() = m;
        return st;
    };
    if (M < 0 || N < 0 || K < 0 || !C || (K > 0 && (!A || !B)))
        return fail(RSRR_EINVAL, "bad argument");
    const int64_t rowsA = conjA ? K : M;
    if (ldc < std::max(1, M) || ldb < std::max(1, K) || lda < std::max<int64_t>(1, rowsA))
        return fail(RSRR_EINVAL, "leading dimension too small");
    if (method < RSRR_GEMM_AUTO || method > RSRR_GEMM_OZAKI_MMA) return fail(RSRR_EINVAL, "unknown method");
    if (hermitian && (!conjA || A != B || lda != ldb || M != N || beta != 0.0))
        return fail(RSRR_EINVAL, "hermitian needs conjA, A == B, lda == ldb, M == N, beta == 0");
    cudaStream_t s = (cudaStream_t)stream;
    const double2 *a = reinterpret_cast<const double2 *>(A);
    const double2 *b = reinterpret_cast<const double2 *>(B);
    double2 *c = reinterpret_cast<double2 *>(C);
    const double flops = 8.0 * M * (double)N * K;
    const bool legacy = method == RSRR_GEMM_OZAKI_MMA;
    const bool sliced = method == RSRR_GEMM_OZAKI || legacy ||
                        (method == RSRR_GEMM_AUTO && flops >= 1073741824.0);
    cudaError_t e;
    if (!sliced) {
        if ((e = fp64_gemm(M, N, K, conjA != 0, a, lda, b, ldb, c, ldc, alpha, beta, s)) != cudaSuccess)
            return fail(RSRR_ECUDA, "fp64 gemm", e);
    } else {
        size_t need = ozaki_workspace_bytes(M, N, K, hermitian != 0);
        if (max_ws_bytes > 0) need = std::min(need, max_ws_bytes);
        // the call's own status word (bounded waits that ran out) follows the
        // slices in the same allocation
        const size_t ws_bytes = need / 256 * 256;
        ZgemmWs hold(s);
        if ((e = hold.get(ws_bytes + 256)) != cudaSuccess) return fail(RSRR_ENOMEM, "work space", e);
        void *ws = hold.p;
        unsigned int *status = reinterpret_cast<unsigned int *>(static_cast<char *>(ws) + ws_bytes);
        unsigned int tmo = 0;
        e = cudaMemsetAsync(status, 0, sizeof(unsigned int), s);
        if (e == cudaSuccess)
            e = ozaki_zgemm(M, N, K, conjA != 0, a, lda, b, ldb, c, ldc, alpha, beta, hermitian != 0, ws,
                            ws_bytes, s, nullptr, nullptr, nullptr, legacy, status);
        if (e == cudaSuccess) e = cudaMemcpyAsync(&tmo, status, sizeof tmo, cudaMemcpyDeviceToHost, s);
        if (e == cudaSuccess) e = cudaStreamSynchronize(s);
        if (e == cudaSuccess && tmo != 0) return fail(RSRR_ETIMEOUT, "a bounded tensor-core wait ran out");
        cudaError_t e2 = cudaStreamSynchronize(s);
        if (e == cudaErrorMemoryAllocation) return fail(RSRR_ENOMEM, "work space below one chunk");
        if (e != cudaSuccess) return fail(RSRR_ECUDA, "sliced gemm", e);
        if (e2 != cudaSuccess) return fail(RSRR_ECUDA, "sync", e2);
    }
    if ((e = cudaStreamSynchronize(s)) != cudaSuccess) return fail(RSRR_ECUDA, "sync", e);
    thread_error().clear();
    return RSRR_OK;
}

extern "C" rsrr_status rsrr_check_wait_timeout(int32_t tries, void *stream) {
    using namespace rsrr;
    auto fail = [](rsrr_status st, const char *msg, cudaError_t e = cudaSuccess) {
        thread_error() = e == cudaSuccess ? std::string(msg) : std::string(msg) + ": " + cudaGetErrorString(e);
        return st;
    };
    if (tries < 1 || tries > (1 << 20)) return fail(RSRR_EINVAL, "rsrr_check_wait_timeout: tries out of range");
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    unsigned int *status = nullptr, tmo = 0;
    cudaError_t e = cudaStreamSynchronize(s);
    if (e == cudaSuccess) e = cudaMalloc(&status, sizeof(unsigned int));
    if (e != cudaSuccess) return fail(RSRR_ECUDA, "rsrr_check_wait_timeout", e);
    e = cudaMemsetAsync(status, 0, sizeof(unsigned int), s);
    if (e == cudaSuccess) {
        ozt_wait_check_kernel<<<1, 32, 0, s>>>((long long)tries, status);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaMemcpyAsync(&tmo, status, sizeof tmo, cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    cudaFree(status);
    if (e != cudaSuccess) return fail(RSRR_ECUDA, "rsrr_check_wait_timeout", e);
    if (tmo == 0) return fail(RSRR_OK, "rsrr_check_wait_timeout: the wait did not run out");
    return fail(RSRR_ETIMEOUT, "a bounded tensor-core wait ran out");
}
