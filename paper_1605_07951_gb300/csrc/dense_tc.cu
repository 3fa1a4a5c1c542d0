// Trailing update of the batched dense complex64 LU on the 5th-generation
// tensor cores (RSRR step 2, Section 4.3: the factorisation of every T(z_j)).
//
// For the panel at column k0 (width jb <= 32) of every point, A22 -= L21 U12
// with L21 = rows k0+jb.. of columns k0..k0+jb-1, U12 = rows k0..k0+jb-1 of
// columns k0+jb.., A22 the trailing block; all three live in the point's
// column-major n x n complex64 matrix.
//
// Complex as one real product (the real embedding):
//   [Cr | Ci] = [Ar | Ai] [[Br, Bi], [-Bi, Br]]
// so a 128 x 128 complex output tile is a 128 x 256 real tile of depth
// K' = 64 (2 jb, zero-padded).  FP32 operands are split into TF32 parts,
// a = a_hi + a_lo (a_hi = a rounded to TF32, a_lo = the rest rounded to
// TF32), and the product is accumulated in FP32 in tensor memory as
// a_lo b_hi + a_hi b_lo + a_hi b_hi (the "3xTF32" scheme: close to FP32
// accuracy, which the FP64 refinement of the samples expects of a complex64
// factor).  Per K-step of 8 the elected thread issues three
// tcgen05.mma.kind::tf32 (M = 128, N = 256); 24 per tile.
//
// Operands are packed by all threads from global memory (L2: the panel and
// the U12 rows are read by every tile of their row / column) into shared
// memory in the K-major core-matrix layout without swizzle: per K-column of
// core matrices (4 TF32 = 16 bytes), all rows contiguous at 16 bytes a row,
// so the descriptor's SBO (next 8-row group) is 128 bytes and its LBO (next
// core matrix along K) 16 x rows bytes.  The accumulator occupies 256 columns
// of tensor memory; the epilogue reads it back (tcgen05.ld) and subtracts it
// from A22, each warp a 32-row slice (its TMEM lanes) of one half of the
// columns, a warp's 32 rows contiguous in memory for every column.
//
// Bound by memory: a tile reads and writes 128 KB of A22 for 24 MMAs.  One CTA fills
// an SM's shared memory, so nothing overlaps but what it issues itself.  It takes tiles
// in turn (a CTA a tile spent 10 000 of 28 000 cycles between CTAs, waiting for its
// stores to leave), all loads, half of A22's included, go out first, and the packing
// behind them stores 16 bytes (4 of K') a lane with the eight lanes of a store phase on
// consecutive rows (one element at a time, eight lanes met in a bank).  All updates of
// 32 points of order 2048: 19.0 -> 10.0 ms; their 46 GB take 6.8 ms at copy rate.
// The one mbarrier wait is bounded; a wait that runs out is counted in the
// caller's status word and the tile is left unchanged.
#include <algorithm>

#include "common.cuh"
#include "rsrr_internal.h"

namespace rsrr {
namespace tc {

constexpr int BM = 128;              // complex rows of a tile
constexpr int BN = 128;              // complex columns of a tile
constexpr int KR = 64;               // real depth (2 x 32)
constexpr int THREADS = 256;
static_assert(BM == BN && (BM * 32) % THREADS == 0, "packing: equal A and B element counts per thread");
constexpr int A_BYTES = BM * KR * 4;           // one TF32 part of A' (32 KB)
constexpr int B_BYTES = 2 * BN * KR * 4;       // one TF32 part of B' (64 KB)
constexpr size_t SMEM = 2 * (size_t)A_BYTES + 2 * (size_t)B_BYTES + 64;
constexpr uint32_t LBO_A = BM * 16;            // next core matrix along K (A')
constexpr uint32_t LBO_B = 2 * BN * 16;        // next core matrix along K (B')
constexpr long long WAIT_LIMIT = 1LL << 22;

// shared-memory matrix descriptor: K-major, no swizzle, start / LBO / SBO in
// 16-byte units, SBO = 128 bytes (next 8-row group), version 1
RSRR_DEV uint64_t smem_desc(uint32_t saddr, uint32_t lbo) {
    return (uint64_t)((saddr >> 4) & 0x3FFF) | ((uint64_t)((lbo >> 4) & 0x3FFF) << 16) |
           ((uint64_t)((128u >> 4) & 0x3FFF) << 32) | (1ull << 46);
}
// instruction descriptor: TF32 x TF32 -> F32, both K-major, M = 128, N = 256
RSRR_DEV uint32_t idesc_tf32_m128_n256() {
    return (1u << 4) | (2u << 7) | (2u << 10) | ((uint32_t)(256 >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
}
RSRR_DEV void mma_tf32(uint32_t d_tmem, uint64_t a, uint64_t b, uint32_t idesc, uint32_t accumulate) {
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
                 "tcgen05.mma.cta_group::1.kind::tf32 [%0], %1, %2, %3, p;\n\t}\n"
                 ::"r"(d_tmem), "l"(a), "l"(b), "r"(idesc), "r"(accumulate) : "memory");
}
RSRR_DEV void commit(uint32_t mbar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n"
                 ::"r"(mbar) : "memory");
}
RSRR_DEV bool wait_parity(uint32_t mbar, uint32_t parity) {
    for (long long it = 0; it < WAIT_LIMIT; ++it) {
        uint32_t done;
        asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
                     "selp.u32 %0, 1, 0, p;\n\t}\n" : "=r"(done) : "r"(mbar), "r"(parity) : "memory");
        if (done) return true;
    }
    return false;
}
RSRR_DEV void tmem_ld16(uint32_t taddr, float (&v)[16]) {
    uint32_t r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];\n"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
#pragma unroll
    for (int j = 0; j < 16; ++j) v[j] = __uint_as_float(r[j]);
}
// a = hi + lo, both TF32 (round to nearest, ties away)
RSRR_DEV void split_tf32(float a, float &hi, float &lo) {
    uint32_t h, l;
    asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(h) : "f"(a));
    hi = __uint_as_float(h);
    asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(l) : "f"(a - hi));
    lo = __uint_as_float(l);
}
// byte offset of element (row, k) of a K-major operand with `rows` rows
RSRR_DEV uint32_t kmajor_off(int row, int k, int rows) {
    return (uint32_t)((k >> 2) * rows * 16 + row * 16 + (k & 3) * 4);
}

__global__ void __launch_bounds__(THREADS, 1)
dense_tc_update_kernel(float2 *__restrict__ A_all, int n, int k0, int jb, int nrt, int64_t tiles,
                       unsigned int *__restrict__ status) {
    extern __shared__ __align__(1024) unsigned char sm[];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    unsigned char *a_hi = sm, *a_lo = sm + A_BYTES;
    unsigned char *b_hi = sm + 2 * A_BYTES, *b_lo = b_hi + B_BYTES;
    uint64_t *mbar = reinterpret_cast<uint64_t *>(sm + 2 * A_BYTES + 2 * B_BYTES);
    uint32_t *tslot = reinterpret_cast<uint32_t *>(sm + 2 * A_BYTES + 2 * B_BYTES + 16);
    const uint32_t mb = (uint32_t)__cvta_generic_to_shared(mbar);

    if (tid == 0) asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(mb));
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 256;\n"
                     ::"r"((uint32_t)__cvta_generic_to_shared(tslot)));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n");
    }
    // tiles in turn, row tiles first, then column tiles, then points: nrt x nrt a point
    uint32_t tmem = 0, parity = 0;
    for (int64_t tile = blockIdx.x; tile < tiles; tile += gridDim.x, parity ^= 1) {
        const int in = (int)(tile % ((int64_t)nrt * nrt));
        float2 *A = A_all + (size_t)(tile / ((int64_t)nrt * nrt)) * n * n;
        const int r0 = k0 + jb + in % nrt * BM;   // first row of the tile
        const int c0 = k0 + jb + in / nrt * BN;   // first column of the tile
        // every load first: the tile's own columns after the operands'
        constexpr int PER = BM * 8 / THREADS;  // groups of 4 depths of A (and of B) per thread
        float2 va[PER][4], vb[PER][4];
        auto b_col = [](int e) { return (e & 7) + 8 * ((e >> 5) & 15); };
        auto b_dep = [](int e) { return ((e >> 3) & 3) + 4 * (e >> 9); };
#pragma unroll
        for (int q = 0; q < PER; ++q) {
            const int e = tid + q * THREADS;
            const int r = r0 + e % BM, c = c0 + b_col(e);
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int t = 4 * (e / BM) + u, tb = 4 * b_dep(e) + u;
                va[q][u] = (t < jb && r < n) ? A[(size_t)(k0 + t) * n + r] : make_float2(0.f, 0.f);
                vb[q][u] = (tb < jb && c < n) ? A[(size_t)c * n + k0 + tb] : make_float2(0.f, 0.f);
            }
        }
        // this thread's part of the tile: a row, 64 columns
        const int cbase = 64 * (warp >> 2), row = r0 + 32 * (warp & 3) + lane;
        float2 cv[64];
        const int cols = row < n ? n - c0 - cbase : 0;  // columns of it that exist
        auto load_columns = [&](int j0) {
            const float2 *p = A + (size_t)(c0 + cbase + j0) * n + row;
#pragma unroll
            for (int j = j0; j < j0 + 32; ++j) {
                cv[j] = j < cols ? *p : make_float2(0.f, 0.f);
                p += n;
            }
        };
        load_columns(0);
        // A' = [Ar | Ai]: row r, depth t (real part) and 32 + t (imaginary part)
        struct Split4 {
            float4 hi, lo;
        };
        auto split4 = [](float x, float y, float z, float w) {
            Split4 f;
            split_tf32(x, f.hi.x, f.lo.x);
            split_tf32(y, f.hi.y, f.lo.y);
            split_tf32(z, f.hi.z, f.lo.z);
            split_tf32(w, f.hi.w, f.lo.w);
            return f;
        };
        auto neg4 = [](float4 v) { return make_float4(-v.x, -v.y, -v.z, -v.w); };
#pragma unroll
        for (int q = 0; q < PER; ++q) {
            const int e = tid + q * THREADS;
            const int r = e % BM, t = 4 * (e / BM);
            const Split4 re = split4(va[q][0].x, va[q][1].x, va[q][2].x, va[q][3].x);
            const Split4 im = split4(va[q][0].y, va[q][1].y, va[q][2].y, va[q][3].y);
            *reinterpret_cast<float4 *>(a_hi + kmajor_off(r, t, BM)) = re.hi;
            *reinterpret_cast<float4 *>(a_lo + kmajor_off(r, t, BM)) = re.lo;
            *reinterpret_cast<float4 *>(a_hi + kmajor_off(r, 32 + t, BM)) = im.hi;
            *reinterpret_cast<float4 *>(a_lo + kmajor_off(r, 32 + t, BM)) = im.lo;
        }
        // B' rows j (real output columns) and BN + j (imaginary): depth t carries
        // (Br, Bi), depth 32 + t carries (-Bi, Br)
#pragma unroll
        for (int q = 0; q < PER; ++q) {
            const int e = tid + q * THREADS;
            const int j = b_col(e), t = 4 * b_dep(e);
            const Split4 re = split4(vb[q][0].x, vb[q][1].x, vb[q][2].x, vb[q][3].x);
            const Split4 im = split4(vb[q][0].y, vb[q][1].y, vb[q][2].y, vb[q][3].y);
            *reinterpret_cast<float4 *>(b_hi + kmajor_off(j, t, 2 * BN)) = re.hi;
            *reinterpret_cast<float4 *>(b_lo + kmajor_off(j, t, 2 * BN)) = re.lo;
            *reinterpret_cast<float4 *>(b_hi + kmajor_off(j, 32 + t, 2 * BN)) = neg4(im.hi);
            *reinterpret_cast<float4 *>(b_lo + kmajor_off(j, 32 + t, 2 * BN)) = neg4(im.lo);
            *reinterpret_cast<float4 *>(b_hi + kmajor_off(BN + j, t, 2 * BN)) = im.hi;
            *reinterpret_cast<float4 *>(b_lo + kmajor_off(BN + j, t, 2 * BN)) = im.lo;
            *reinterpret_cast<float4 *>(b_hi + kmajor_off(BN + j, 32 + t, 2 * BN)) = re.hi;
            *reinterpret_cast<float4 *>(b_lo + kmajor_off(BN + j, 32 + t, 2 * BN)) = re.lo;
        }
        asm volatile("" ::: "memory");  // not before the registers of va and vb are free
        load_columns(32);
        // the packed operands become visible to the tensor core (async proxy)
        asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
        asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
        __syncthreads();
        asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
        tmem = *tslot;
        if (tid == 0) {
            const uint32_t idesc = idesc_tf32_m128_n256();
            const uint32_t ah = (uint32_t)__cvta_generic_to_shared(a_hi), al = (uint32_t)__cvta_generic_to_shared(a_lo);
            const uint32_t bh = (uint32_t)__cvta_generic_to_shared(b_hi), bl = (uint32_t)__cvta_generic_to_shared(b_lo);
#pragma unroll 1
            for (int kk = 0; kk < KR / 8; ++kk) {
                const uint32_t ao = (uint32_t)(kk * 2) * LBO_A, bo = (uint32_t)(kk * 2) * LBO_B;
                mma_tf32(tmem, smem_desc(al + ao, LBO_A), smem_desc(bh + bo, LBO_B), idesc, kk > 0 ? 1u : 0u);
                mma_tf32(tmem, smem_desc(ah + ao, LBO_A), smem_desc(bl + bo, LBO_B), idesc, 1u);
                mma_tf32(tmem, smem_desc(ah + ao, LBO_A), smem_desc(bh + bo, LBO_B), idesc, 1u);
            }
            commit(mb);
        }
        __syncwarp();
        // epilogue: warp w reads TMEM lanes 32 (w % 4) .. (its 32 rows) for the
        // complex columns 64 (w / 4) .. +63: real parts in TMEM columns j, imaginary
        // parts in columns BN + j
        const uint32_t trow = tmem + ((uint32_t)(32 * (warp & 3)) << 16);
        const bool ok = wait_parity(mb, parity);
        asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
        float2 *out = A + (size_t)(c0 + cbase) * n + row;
        asm volatile("" : "+l"(out));  // its 64 addresses are not kept from the loads
#pragma unroll
        for (int q = 0; q < 64; q += 16) {
            float re[16], im[16];
            tmem_ld16(trow + (uint32_t)(cbase + q), re);
            tmem_ld16(trow + (uint32_t)(BN + cbase + q), im);
#pragma unroll
            for (int j = 0; j < 16; ++j) {
                if (ok && q + j < cols) *out = make_float2(cv[q + j].x - re[j], cv[q + j].y - im[j]);
                out += n;
            }
        }
        if (!ok && lane == 0) atomicAdd(status, 1u);
        if (!__syncthreads_and(ok)) break;  // no further tile on this SM
    }
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 256;\n" ::"r"(tmem));
}

}  // namespace tc

cudaError_t launch_dense_tc_update(float2 *A, int n, int k0, int jb, int N, unsigned int *status,
                                   cudaStream_t s) {
    const int rest = n - k0 - jb;
    if (rest <= 0) return cudaSuccess;
    if (jb > 32 || !status) return cudaErrorInvalidValue;
    cudaError_t e = cudaFuncSetAttribute(tc::dense_tc_update_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)tc::SMEM);
    if (e != cudaSuccess) return e;
    int dev = 0, nsm = 152;
    if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
    if ((e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
    const int nrt = (rest + tc::BM - 1) / tc::BM;
    const int64_t tiles = (int64_t)nrt * nrt * N;
    tc::dense_tc_update_kernel<<<(unsigned)std::min<int64_t>(tiles, nsm), tc::THREADS, tc::SMEM, s>>>(A, n, k0, jb, nrt,
                                                                                                    tiles, status);
    return cudaGetLastError();
}

}  // namespace rsrr
