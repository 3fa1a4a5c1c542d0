// Moments of SS-FULL (Section 3.3 with U = I) for the projected NEP on the
// GPU, in FP64:
//
//     A_alpha = sum_q w_q s_q^alpha T_Q(z_q)^{-1},   alpha < 2 K_Q,
//
// with the N_Q trapezoid nodes z_q = gamma + a cos t_q + i b sin t_q,
// t_q = 2 pi (q + 1/2) / N_Q, weights w_q = (-a sin t_q + i b cos t_q) / N_Q
// (Section 5.1) and scaled powers s_q = (z_q - gamma) / rho, rho = max(a, b).
// Nodes are processed in chunks: T_Q(z_q) = sum_i f_i(z_q) P_i is assembled
// for every node of the chunk, factored by the batched complex128 dense LU
// (partial pivoting), inverted, and the weighted inverses summed into the
// moments in a fixed node order.  For symmetric real A_i and f_i with
// f_i(conj z) = conj f_i(z), T_Q(conj z) = T_Q(z)^H: on a contour symmetric
// about the real axis only one node of each conjugate pair is factored, half
// of the work (bound by the FP64 unit).  The Hankel SVD and the small eigenproblem stay on the
// host (ssfull_host.cpp).
#include <algorithm>
#include <cmath>
#include <complex>
#include <vector>

#include "common.cuh"
#include "rsrr_handle.h"

namespace rsrr {

// T[b] = sum_i f[b][i] P_i for the nodes of a chunk (k x k each)
__global__ void tq_assemble_kernel(double2 *__restrict__ T, const double2 *__restrict__ P,
                                   const double2 *__restrict__ f, int m, int64_t kk) {
    const int b = blockIdx.y;
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < kk;
         e += (int64_t)gridDim.x * blockDim.x) {
        double2 acc = make_double2(0.0, 0.0);
        for (int i = 0; i < m; ++i) acc = cfma(acc, f[(size_t)b * m + i], P[(size_t)i * kk + e]);
        T[(size_t)b * kk + e] = acc;
    }
}

// Acc[alpha] += sum_b c[b][alpha] F[b] + d[b][alpha] F[b]^H, nodes summed in
// order.  A block of 256 threads owns a 16 x 16 tile; the mirrored tile it needs
// for F^H comes through shared memory (mirror = 0: d is zero and not read).
__global__ void __launch_bounds__(256)
tq_moment_kernel(double2 *__restrict__ Acc, const double2 *__restrict__ F, const double2 *__restrict__ c,
                 const double2 *__restrict__ d, int nb, int nmom, int k, int mirror) {
    __shared__ double2 s_t[16][17];
    const int tx = threadIdx.x % 16, ty = threadIdx.x / 16;
    const int i = blockIdx.x * 16 + tx, j = blockIdx.y * 16 + ty;        // this thread's element
    const int mi = blockIdx.y * 16 + tx, mj = blockIdx.x * 16 + ty;      // its part of the mirrored tile
    const bool in = i < k && j < k, min = mi < k && mj < k;
    const size_t kk = (size_t)k * k, e = (size_t)j * k + i, me = (size_t)mj * k + mi;
    for (int al0 = 0; al0 < nmom; al0 += 4) {
        double2 acc[4];
#pragma unroll
        for (int a = 0; a < 4; ++a)
            acc[a] = in && al0 + a < nmom ? Acc[(al0 + a) * kk + e] : make_double2(0.0, 0.0);
        for (int b = 0; b < nb; ++b) {
            const double2 f = in ? F[b * kk + e] : make_double2(0.0, 0.0);
            double2 h = make_double2(0.0, 0.0);
            if (mirror) {
                __syncthreads();
                s_t[ty][tx] = min ? F[b * kk + me] : make_double2(0.0, 0.0);
                __syncthreads();
                h = s_t[tx][ty];
                h.y = -h.y;
            }
#pragma unroll
            for (int a = 0; a < 4; ++a) {
                if (al0 + a >= nmom) break;
                acc[a] = cfma(acc[a], c[(size_t)b * nmom + al0 + a], f);
                if (mirror) acc[a] = cfma(acc[a], d[(size_t)b * nmom + al0 + a], h);
            }
        }
#pragma unroll
        for (int a = 0; a < 4; ++a)
            if (in && al0 + a < nmom) Acc[(al0 + a) * kk + e] = acc[a];
    }
}

static int grid_cap(int64_t work, int threads, int cap) {
    return (int)std::max<int64_t>(1, std::min<int64_t>((work + threads - 1) / threads, cap));
}

// node chunk size: T and F of the chunk within `bytes`, at most NQ
static int ssfull_chunk(int64_t k, int NQ, size_t bytes) {
    const size_t per = sizeof(double2) * (size_t)k * k * 2;
    return (int)std::max<size_t>(1, std::min<size_t>(NQ, bytes / std::max<size_t>(per, 1)));
}

// device bytes of the moment stage for basis size k
size_t ssfull_dev_bytes(int64_t k, int m, int NQ, int KQ) {
    const size_t B = ssfull_chunk(k, NQ, kSsfullChunkBytes);
    const size_t kk = (size_t)k * k;
    const size_t nblk = ((size_t)k + NB_C128 - 1) / NB_C128;
    return sizeof(double2) * (2 * B * kk + (size_t)2 * KQ * kk + B * (m + 4 * KQ) +
                              B * nblk * 2 * NB_C128 * NB_C128) +
           sizeof(int32_t) * (B * k + B) + 9 * 256;
}

rsrr_status Handle::ssfull_moments(const std::vector<std::complex<double>> &fq,
                                   const std::vector<std::complex<double>> &zq,
                                   const std::vector<std::complex<double>> &wq, int KQ,
                                   std::vector<std::vector<std::complex<double>>> &Am) {
    using cplx = std::complex<double>;
    cudaStream_t s = hs;
    const int NQ = (int)zq.size();
    const int nmom = 2 * KQ;
    const int64_t kk = (int64_t)k * k;
    const int B = ssfull_chunk(k, NQ, kSsfullChunkBytes);
    const size_t nblk = ((size_t)k + NB_C128 - 1) / NB_C128;
    const size_t bytes = ssfull_dev_bytes(k, m, NQ, KQ);
    void *buf = nullptr;
    cudaError_t e = pool ? cudaMallocFromPoolAsync(&buf, bytes, pool, s) : cudaMalloc(&buf, bytes);
    if (e != cudaSuccess) return fail(RSRR_ENOMEM, "SS-FULL moment buffers", e);
    struct Free {
        Handle *h;
        void *p;
        ~Free() { h->raw_free(p); }
    } guard{this, buf};
    char *p = static_cast<char *>(buf);
    auto take = [&p](size_t b) {
        char *q = p;
        p += (b + 255) / 256 * 256;
        return q;
    };
    double2 *dT = reinterpret_cast<double2 *>(take(sizeof(double2) * B * kk));
    double2 *dF = reinterpret_cast<double2 *>(take(sizeof(double2) * B * kk));
    double2 *dA = reinterpret_cast<double2 *>(take(sizeof(double2) * nmom * kk));
    double2 *df = reinterpret_cast<double2 *>(take(sizeof(double2) * B * m));
    double2 *dc = reinterpret_cast<double2 *>(take(sizeof(double2) * B * nmom));
    double2 *dd = reinterpret_cast<double2 *>(take(sizeof(double2) * B * nmom));
    double2 *dinv = reinterpret_cast<double2 *>(take(sizeof(double2) * B * nblk * 2 * NB_C128 * NB_C128));
    int32_t *dpiv = reinterpret_cast<int32_t *>(take(sizeof(int32_t) * B * k));
    int32_t *dinfo = reinterpret_cast<int32_t *>(take(sizeof(int32_t) * B));
    if ((size_t)(p - static_cast<char *>(buf)) > bytes) return fail(RSRR_ESTATE, "SS-FULL buffer layout");

    const double rho = std::max(region.a, region.b);
    const cplx gamma(region.center.re, region.center.im);
    // nodes to factor: all, or one of each conjugate pair (q, NQ - 1 - q); the
    // pair's values agree to rounding or the symmetry is not used
    bool paired = sym_real;
    auto conj_close = [](cplx a, cplx b) { return std::abs(a - std::conj(b)) <= 16.0 * 2.2204460492503131e-16 * std::abs(b); };
    for (int q = 0; q < NQ && paired; ++q) {
        const int r = NQ - 1 - q;
        paired = conj_close(zq[r], zq[q]);
        for (int i = 0; i < m && paired; ++i) paired = conj_close(fq[(size_t)r * m + i], fq[(size_t)q * m + i]);
    }
    const int nodes = paired ? (NQ + 1) / 2 : NQ;
    std::vector<double2> hf((size_t)B * m), hc((size_t)B * nmom), hd((size_t)B * nmom);
    std::vector<int32_t> info(B);
    if ((e = cudaMemsetAsync(dA, 0, sizeof(double2) * nmom * kk, s)) != cudaSuccess)
        return fail(RSRR_ECUDA, "memset", e);
    for (int q0 = 0; q0 < nodes; q0 += B) {
        const int nb = std::min(B, nodes - q0);
        for (int bq = 0; bq < nb; ++bq) {
            const int q = q0 + bq;
            for (int i = 0; i < m; ++i) {
                const cplx v = fq[(size_t)q * m + i];
                hf[(size_t)bq * m + i] = make_double2(v.real(), v.imag());
            }
            auto powers = [&](int node, std::vector<double2> &out) {
                const cplx sz = (zq[node] - gamma) / rho;
                cplx c = wq[node];
                for (int al = 0; al < nmom; ++al) {
                    out[(size_t)bq * nmom + al] = make_double2(c.real(), c.imag());
                    c *= sz;
                }
            };
            powers(q, hc);
            if (paired && NQ - 1 - q != q) powers(NQ - 1 - q, hd);
            else std::fill(hd.begin() + (size_t)bq * nmom, hd.begin() + (size_t)(bq + 1) * nmom, make_double2(0.0, 0.0));
        }
        // (pageable sources: each copy returns once staged, so hf, hc, hd may be refilled)
        if ((e = cudaMemcpyAsync(df, hf.data(), sizeof(double2) * nb * m, cudaMemcpyHostToDevice, s)) !=
                cudaSuccess ||
            (e = cudaMemcpyAsync(dc, hc.data(), sizeof(double2) * nb * nmom, cudaMemcpyHostToDevice, s)) !=
                cudaSuccess ||
            (e = cudaMemcpyAsync(dd, hd.data(), sizeof(double2) * nb * nmom, cudaMemcpyHostToDevice, s)) !=
                cudaSuccess)
            return fail(RSRR_ECUDA, "SS-FULL coefficients", e);
        tq_assemble_kernel<<<dim3(grid_cap(kk, 256, 1024), nb), 256, 0, s>>>(dT, d_P, df, m, kk);
        if ((e = cudaGetLastError()) != cudaSuccess) return fail(RSRR_ECUDA, "SS-FULL assemble", e);
        if ((e = launch_dense_lu_c128(dT, dpiv, dinfo, dinv, k, nb, s, &launches)) != cudaSuccess)
            return fail(RSRR_ECUDA, "SS-FULL LU", e);
        if ((e = launch_dense_inverse_c128(dT, dpiv, dinv, dF, k, nb, s)) != cudaSuccess)
            return fail(RSRR_ECUDA, "SS-FULL inverse", e);
        const unsigned tiles = (unsigned)((k + 15) / 16);
        tq_moment_kernel<<<dim3(tiles, tiles), 256, 0, s>>>(dA, dF, dc, dd, nb, nmom, k, paired ? 1 : 0);
        if ((e = cudaGetLastError()) != cudaSuccess) return fail(RSRR_ECUDA, "SS-FULL moments", e);
        if ((e = cudaMemcpyAsync(info.data(), dinfo, sizeof(int32_t) * nb, cudaMemcpyDeviceToHost, s)) !=
                cudaSuccess ||
            (e = cudaStreamSynchronize(s)) != cudaSuccess)
            return fail(RSRR_ECUDA, "SS-FULL chunk", e);
        launches += 3;
        for (int bq = 0; bq < nb; ++bq)
            if (info[bq] != 0)
                return fail(RSRR_ESINGULAR, "rsrr_solve: projected T_Q singular at a quadrature node");
    }
    Am.assign(nmom, std::vector<cplx>(kk));
    for (int al = 0; al < nmom; ++al)
        if ((e = cudaMemcpyAsync(Am[al].data(), dA + (size_t)al * kk, sizeof(double2) * kk,
                                 cudaMemcpyDeviceToHost, s)) != cudaSuccess)
            return fail(RSRR_ECUDA, "SS-FULL moments to host", e);
    if ((e = cudaStreamSynchronize(s)) != cudaSuccess) return fail(RSRR_ECUDA, "SS-FULL sync", e);
    return RSRR_OK;
}

}  // namespace rsrr
