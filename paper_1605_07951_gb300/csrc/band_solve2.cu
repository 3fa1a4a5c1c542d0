// Streaming banded solve with the factors of band_lu_kernel: X = (P L U)^{-1} B
// for every sampling point (Section 4.3's X_j = T(z_j)^{-1} U), one CTA per
// (point, chunk of LC right-hand sides).
//
// Forward, block by block (NB rows): the block's composed row permutation
// (precomputed by block_perm_kernel as (position, source) pairs; usually
// none) is applied to the shared-memory window, y = L11^{-1} (P b)_top, and the
// rows below are updated, b_below -= L21 y.  Backward, from the last block:
// x = U11^{-1} y_block, then the rows above are updated, y_above -= U_above x
// (the same column-panel form as the forward pass), from the first row that
// reaches the block's columns on (ku rows above without interchanges, at
// most kl + ku).
//
// The factor panels (L21 below / U above a block, one contiguous run per column
// in the band layout) stream through a ring of shared-memory slots.  A slot
// has its own producer warps: they wait until it is free, copy one unit (up
// to rc panel rows of one block; with a block's first unit its diagonal-block
// inverse and its permutation record) by cp.async, wait for their copies and
// hand it over; both hand-overs are named barriers, so nothing spins.  Runs
// start at any element: each column copies the 16-byte-aligned superset and
// reads from its offset.  The other warps only compute: two block
// barriers a step, the rows that enter the window loaded a step ahead.
//
// What bounds it: the chain of dependent block steps.  With the copies issued
// by the computing warps themselves, kl + ku rows above every block and four
// barriers a step, the full-size problem (n = 40000, half-bandwidth 200, 64
// points, 32 right-hand sides) took 21.2 ms a solve; now 11.1 ms, of which 6 ms
// are FP32 FMAs (16 right-hand sides a CTA: 128 CTAs).  Sweeps of two points 9.6 ->
// 4.8 ms; half-bandwidth 61, n = 3721, 32 points 0.53 -> 0.30 ms; complex128,
// half-bandwidth 70, n = 4900 12.5 -> 4.5 ms (more CTAs for few points, too).
#include <algorithm>
#include <cstdint>

#include "common.cuh"
#include "rsrr_internal.h"

namespace rsrr {

constexpr int SV_PRODUCERS = 256;  // threads that copy, split evenly over the slots
constexpr int SV_BAR = 1, SV_FULL = 2, SV_EMPTY = 6;  // named barriers (one per slot from the last two on)

// ---------------------------------------------------------------------------
// Per block of NB rows: the composed permutation (the LU swaps row j0+cc with
// piv[j0+cc] for cc = 0..jb-1 in order; position r of the block's window, rows
// j0 .. j0+pr-1, then holds original row j0 + perm[r]) as (r << 16) | perm[r]
// for every r with perm[r] != r; then their number; then the first row of U
// that reaches the block's columns: the smallest i with piv[i] + ku >= j0 (a
// row's last column is the largest piv[i'] + ku over i' <= i).  One warp per
// (point, block).
// ---------------------------------------------------------------------------
constexpr int BP_WARPS = 8;
constexpr int BP_MAXR = KL_MAX + 32;

__global__ void block_perm_kernel(int32_t *__restrict__ bperm, const int32_t *__restrict__ piv_all,
                                  int n, int kl, int ku, int NB, int nblk, int N) {
    __shared__ int sp[BP_WARPS][BP_MAXR];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int64_t total = (int64_t)N * nblk;
    for (int64_t task = (int64_t)blockIdx.x * BP_WARPS + w; task < total;
         task += (int64_t)gridDim.x * BP_WARPS) {
        const int pt = (int)(task / nblk), j = (int)(task % nblk);
        const int j0 = j * NB;
        const int jb = min(NB, n - j0);
        const int pr = min(n - j0, jb + kl);
        const int32_t *piv = piv_all + (size_t)pt * n;
        int *perm = sp[w];
        for (int r = lane; r < pr; r += 32) perm[r] = r;
        __syncwarp();
        const int own = lane < jb ? piv[j0 + lane] - j0 : lane;  // NB <= 32: a pivot per lane
        for (int cc = 0; cc < jb; ++cc) {
            int p = __shfl_sync(0xffffffffu, own, cc);
            if (p <= cc || p >= pr) continue;  // (out-of-range pivots never come from the LU)
            if (lane == 0) {
                const int t = perm[cc];
                perm[cc] = perm[p];
                perm[p] = t;
            }
        }
        __syncwarp();
        int32_t *out = bperm + (size_t)task * bp_ints(NB);
        int cnt = 0;
        for (int r0 = 0; r0 < pr; r0 += 32) {
            const int r = r0 + lane;
            const bool moved = r < pr && perm[r] != r;
            const unsigned m = __ballot_sync(0xffffffffu, moved);
            const int pos = cnt + __popc(m & ((1u << lane) - 1u));
            if (moved && pos < 2 * NB) out[pos] = (r << 16) | perm[r];
            cnt += __popc(m);
        }
        int top = j0;
        for (int i0 = max(0, j0 - kl - ku); i0 < j0; i0 += 32) {
            const int i = i0 + lane;
            const unsigned m = __ballot_sync(0xffffffffu, i < j0 && piv[min(i, n - 1)] + ku >= j0);
            if (m) {
                top = i0 + __ffs(m) - 1;
                break;
            }
        }
        if (lane == 0) {
            out[2 * NB] = min(cnt, 2 * NB);
            out[2 * NB + 1] = top;
        }
        __syncwarp();
    }
}

// ---------------------------------------------------------------------------
RSRR_DEV void sv_copy16(unsigned saddr, const void *g) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(saddr), "l"(g));
}
RSRR_DEV void sv_sync(int id, int threads) { asm volatile("bar.sync %0, %1;\n" ::"r"(id), "r"(threads) : "memory"); }
RSRR_DEV void sv_arrive(int id, int threads) {
    asm volatile("bar.arrive %0, %1;\n" ::"r"(id), "r"(threads) : "memory");
}

// K adjacent elements of shared memory, in 16-byte accesses where they fill them
// (the address is then a multiple of 16 bytes)
template <int K> RSRR_DEV void sv_get(const float2 *s, float2 (&o)[K]) {
    if constexpr (K % 2 == 0) {
#pragma unroll
        for (int k = 0; k < K; k += 2) {
            const float4 q = *reinterpret_cast<const float4 *>(s + k);
            o[k] = make_float2(q.x, q.y);
            o[k + 1] = make_float2(q.z, q.w);
        }
    } else {
#pragma unroll
        for (int k = 0; k < K; ++k) o[k] = s[k];
    }
}
template <int K> RSRR_DEV void sv_put(float2 *s, const float2 (&o)[K]) {
    if constexpr (K % 2 == 0) {
#pragma unroll
        for (int k = 0; k < K; k += 2)
            *reinterpret_cast<float4 *>(s + k) = make_float4(o[k].x, o[k].y, o[k + 1].x, o[k + 1].y);
    } else {
#pragma unroll
        for (int k = 0; k < K; ++k) s[k] = o[k];
    }
}
template <int K, typename C> RSRR_DEV void sv_get(const C *s, C (&o)[K]) {
#pragma unroll
    for (int k = 0; k < K; ++k) o[k] = s[k];
}
template <int K, typename C> RSRR_DEV void sv_put(C *s, const C (&o)[K]) {
#pragma unroll
    for (int k = 0; k < K; ++k) s[k] = o[k];
}

// shared memory of one CTA: the window of WR rows, the slots, y, gathered rows
template <typename C, int NB, int LC> struct SvLayout {
    static constexpr int E16 = 16 / (int)sizeof(C);  // elements per 16 bytes
    // window row stride: rows of a warp fall in different banks; for 8-byte
    // types a multiple of 16 bytes, so that two right-hand sides move in one access
    static constexpr int WLD = LC + (sizeof(C) == 8 ? 2 : 1);
    static_assert(sizeof(C) != 8 || LC % 2 == 0, "16-byte accesses of two elements");
    static constexpr size_t D_BYTES = sizeof(C) * NB * NB;
    static constexpr size_t P_BYTES = 4 * bp_ints(NB);
    static RSRR_HD size_t w_bytes(int WR) { return ((sizeof(C) * (size_t)WR * WLD + 15) / 16) * 16; }
    static RSRR_HD size_t slot(int rc) { return D_BYTES + P_BYTES + sizeof(C) * NB * (size_t)(rc + E16); }
    static size_t smem(int WR, int rc, int nslot) {
        return w_bytes(WR) + nslot * slot(rc) + sizeof(C) * NB * LC + sizeof(C) * (size_t)(2 * NB) * LC;
    }
};

// CW computing warps; a lane updates RR rows (32 apart) by CG right-hand sides.
template <typename C, int NB, int LC, int CW, int RR, int CG>
__global__ void __launch_bounds__(32 * CW + SV_PRODUCERS, 1)
band_solve_stream_kernel(const C *__restrict__ ab_all, const int32_t *__restrict__ bperm_all,
                         const C *__restrict__ dinv_all, C *__restrict__ B_all, int n, int kl, int ku,
                         int ldab, int L, int WR, int rc, int nslot, const int32_t *__restrict__ skip,
                         const int32_t *__restrict__ gate, int gate_want) {
    using LY = SvLayout<C, NB, LC>;
    // a gated launch runs only if the gate word holds gate_want (one of the
    // shapes of a refinement sweep, chosen on the device)
    if (gate && __ldg(gate) != gate_want) return;
    constexpr int E16 = LY::E16, WLD = LY::WLD, CT = 32 * CW;
    constexpr bool WIDE = sizeof(typename real_of<C>::type) == 8;  // FP64 arithmetic
    const int pt = blockIdx.y;
    if (skip && skip[pt]) return;
    const int col0 = blockIdx.x * LC;
    const int ncol = min(LC, L - col0);
    const int nblk = (n + NB - 1) / NB;
    const int KV = kl + ku;
    const C *ab = ab_all + (size_t)pt * ldab * n;
    const C *dinv = dinv_all + (size_t)pt * nblk * 2 * NB * NB;
    const int32_t *bperm = bperm_all + (size_t)pt * nblk * bp_ints(NB);
    C *B = B_all + (size_t)pt * L * n + (size_t)col0 * n;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;

    extern __shared__ __align__(16) unsigned char sv_smem[];
    C *W = reinterpret_cast<C *>(sv_smem);  // [WR][WLD], row i at i mod WR
    unsigned char *slots = sv_smem + LY::w_bytes(WR);
    const unsigned slot_bytes = (unsigned)LY::slot(rc);
    C *Yb = reinterpret_cast<C *>(slots + nslot * slot_bytes);  // [NB][LC]
    C *Gp = Yb + NB * LC;                                       // [2 NB][LC]
    const int pld = rc + E16;                                   // panel column stride
    const int handover = CT + SV_PRODUCERS / nslot;             // threads of a slot's two barriers

    if (warp >= CW) {
        // ------------------------------------------------------- producers
        const int pwarps = SV_PRODUCERS / 32 / nslot;  // of one slot
        const int pw = warp - CW, mine = pw / pwarps, w = pw % pwarps, pt_tid = w * 32 + lane;
        const unsigned slot = (unsigned)__cvta_generic_to_shared(slots + mine * slot_bytes);
        const unsigned pan = slot + (unsigned)(LY::D_BYTES + LY::P_BYTES);
        const ptrdiff_t hop = (ptrdiff_t)(ldab - 1) * (ptrdiff_t)sizeof(C);  // one column right, same row
        int u = 0;  // slot of the unit at hand
        bool used = false;
        for (int phase = 0; phase < 2; ++phase) {
            int top = phase ? __ldg(&bperm[(size_t)(nblk - 1) * bp_ints(NB) + 2 * NB + 1]) : 0;
            for (int q = 0; q < nblk; ++q) {
                const int j = phase ? nblk - 1 - q : q, j0 = j * NB, jb = min(NB, n - j0);
                const int top_next = phase && j > 0 ? __ldg(&bperm[(size_t)(j - 1) * bp_ints(NB) + 2 * NB + 1]) : 0;
                const int i_lo = phase ? top : j0 + jb;  // first panel row
                const int rows = phase ? j0 - top : min(n - j0, jb + kl) - jb;
                int ra = 0;
                do {
                    if (u == mine) {
                        if (used) sv_sync(SV_EMPTY + mine, handover);
                        used = true;
                        if (ra == 0) {
                            const unsigned char *d = reinterpret_cast<const unsigned char *>(
                                dinv + ((size_t)j * 2 + phase) * NB * NB);
                            for (int o = pt_tid; o < (int)(LY::D_BYTES / 16); o += pwarps * 32)
                                sv_copy16(slot + o * 16, d + o * 16);
                            const unsigned char *b = reinterpret_cast<const unsigned char *>(bperm + (size_t)j * bp_ints(NB));
                            for (int o = pt_tid; o < (int)(LY::P_BYTES / 16); o += pwarps * 32)
                                sv_copy16(slot + (unsigned)LY::D_BYTES + o * 16, b + o * 16);
                        }
                        const int len = min(rc, rows - ra);
                        if (len > 0) {
                            // row i_lo + ra of column j0 + w; the copies start at the 16 bytes it lies in
                            const unsigned char *src = reinterpret_cast<const unsigned char *>(
                                ab + (size_t)j0 * ldab + KV + (i_lo + ra) - j0) + w * hop;
                            unsigned dst = pan + (unsigned)(w * pld * (int)sizeof(C));
                            for (int t = w; t < jb; t += pwarps) {
                                const int off = (int)(reinterpret_cast<uintptr_t>(src) & 15u);
                                const unsigned char *from = src - off + lane * 16;
                                const int bytes = len * (int)sizeof(C) + off;
                                for (int o = lane * 16; o < bytes; o += 512, from += 512) sv_copy16(dst + o, from);
                                src += pwarps * hop;
                                dst += (unsigned)(pwarps * pld * (int)sizeof(C));
                            }
                        }
                        asm volatile("cp.async.commit_group;\ncp.async.wait_group 0;\n" ::: "memory");
                        sv_arrive(SV_FULL + mine, handover);
                    }
                    if (++u == nslot) u = 0;
                    ra += rc;
                } while (ra < rows);
                top = top_next;
            }
        }
        if (used) sv_sync(SV_EMPTY + mine, handover);
        return;
    }

    // ----------------------------------------------------------- consumers
    // this thread's share of the diagonal solve: DC columns of row dr
    constexpr int DC = NB * LC > CT ? NB * LC / CT : 1;
    static_assert(LC % DC == 0 && (NB * LC) % DC == 0, "diagonal solve mapping");
    const int dcol = tid % (LC / DC) * DC, dr = tid / (LC / DC);
    // and of the rows that enter the window
    constexpr int NE = (NB * LC + CT - 1) / CT;
    // position in 16-byte units of the panel value at row i0 of column j0 + t: (pos0 + i0 + t (ldab - 1)) mod E16
    const unsigned pos0 = (unsigned)((reinterpret_cast<uintptr_t>(ab) & 15u) / sizeof(C)) + (unsigned)KV;
    int u = 0;
    for (int phase = 0; phase < 2; ++phase) {
        // the first block's window
        {
            const int jl = (nblk - 1) * NB;
            const int r0 = phase ? max(0, jl - KV) : 0, r1 = phase ? n : min(n, NB + kl);
            for (int r = r0 + (tid & 31); r < r1; r += 32)
                for (int c = tid >> 5; c < LC; c += CW)
                    W[(size_t)(r % WR) * WLD + c] = c < ncol ? B[(size_t)c * n + r] : czero<C>();
        }
        int jb0 = phase ? ((nblk - 1) * NB) % WR : 0;  // window row of the block's first row
        for (int q = 0; q < nblk; ++q) {
            const int j = phase ? nblk - 1 - q : q, j0 = j * NB, jb = min(NB, n - j0);
            const unsigned char *slot = slots + u * slot_bytes;
            // the rows that enter with the next block, loaded a step ahead
            C in[NE];
#pragma unroll
            for (int k = 0; k < NE; ++k) {
                const int e = tid + k * CT, c = e / NB;
                const int r = phase ? j0 - NB - KV + e % NB : j0 + NB + kl + e % NB;
                in[k] = czero<C>();
                if (c < ncol && r >= 0 && r < n) in[k] = B[(size_t)c * n + r];
            }
            sv_sync(SV_FULL + u, handover);  // the unit is here, and every warp is done with the last block
            const C *D = reinterpret_cast<const C *>(slot);
            const int32_t *rec = reinterpret_cast<const int32_t *>(slot + LY::D_BYTES);
            // window row of row j0 + off, -WR <= off < 2 WR - jb0
            auto wrow = [&](int off) {
                const int r = jb0 + off;
                return r >= WR ? r - WR : r < 0 ? r + WR : r;
            };
            if (phase == 0) {
                const int cnt = rec[2 * NB];
                if (cnt > 0) {  // the block's interchanges
                    for (int o = tid; o < cnt * LC; o += CT)
                        Gp[o] = W[wrow(rec[o / LC] & 0xFFFF) * WLD + o % LC];
                    sv_sync(SV_BAR, CT);
                    for (int o = tid; o < cnt * LC; o += CT)
                        W[wrow(rec[o / LC] >> 16) * WLD + o % LC] = Gp[o];
                    sv_sync(SV_BAR, CT);
                }
            }
            // y = L11^{-1} (P b)_top  or  x = U11^{-1} y_block
            if (dr < NB) {
                const C *d = D + dr, *Wb = W + jb0 * WLD + dcol;
                C v[DC];
#pragma unroll
                for (int c = 0; c < DC; ++c) v[c] = czero<C>();
                if (jb == NB) {
#pragma unroll(WIDE ? 4 : NB)
                    for (int t = 0; t < NB; ++t) {
                        const C dt = d[t * NB];
                        C w[DC];
                        sv_get<DC>(Wb + t * WLD, w);
#pragma unroll
                        for (int c = 0; c < DC; ++c) v[c] = cfma(v[c], dt, w[c]);
                    }
                } else {
                    for (int t = 0; t < jb; ++t)
#pragma unroll
                        for (int c = 0; c < DC; ++c) v[c] = cfma(v[c], d[t * NB], Wb[t * WLD + c]);
                }
                sv_put<DC>(Yb + dr * LC + dcol, v);
#pragma unroll
                for (int c = 0; c < DC; ++c)
                    if (dr < jb && dcol + c < ncol) B[(size_t)(dcol + c) * n + j0 + dr] = v[c];
            }
            const int i_lo = phase ? rec[2 * NB + 1] : j0 + jb;
            const int rows = phase ? j0 - i_lo : min(n - j0, jb + kl) - jb;
            sv_sync(SV_BAR, CT);
            // the panel, unit by unit: W[rows] -= P Yb
            int ra = 0;
            for (;;) {
                const C *P = reinterpret_cast<const C *>(slot + LY::D_BYTES + LY::P_BYTES);
                const int len = min(rc, rows - ra);
                const int i0 = i_lo + ra;
                const unsigned o0 = pos0 + (unsigned)j0 * (unsigned)(ldab - 1) + (unsigned)i0, od = (unsigned)(ldab - 1);
                if (len > 0) {
                    if constexpr (WIDE) {
                        // one element a lane: a warp-wide FP64 FMA takes 64 cycles, however many lanes are active
                        for (int e = tid; e < len * LC; e += CT) {
                            const int col = e / len, rr = e - col * len, i = i0 + rr;
                            C *wr = W + wrow(i - j0) * WLD + col;
                            C acc = *wr;
                            const int tm = phase ? min(jb, i + KV - j0 + 1) : jb;
#pragma unroll 4
                            for (int t = 0; t < tm; ++t)
                                acc = cfms(acc, P[t * pld + (int)((o0 + t * od) & (E16 - 1)) + rr], Yb[t * LC + col]);
                            *wr = acc;
                        }
                    } else {
                        // a task: 32 RR rows by CG columns
                        constexpr int CGN = LC / CG;
                        const int tasks = (len + 32 * RR - 1) / (32 * RR) * CGN;
                        for (int task = warp; task < tasks; task += CW) {
                            const int rg = task / CGN * (32 * RR), cg = task % CGN * CG;
                            C acc[RR][CG];
                            C *wr[RR];
#pragma unroll
                            for (int a = 0; a < RR; ++a) {
                                // (a lane past the last row computes what lies behind the panel and stores nothing)
                                wr[a] = W + wrow(i0 - j0 + min(rg + lane + 32 * a, len - 1)) * WLD + cg;
                                sv_get<CG>(wr[a], acc[a]);
                            }
                            const C *y = Yb + cg;
                            // backward: U(i, j0+t) lies in the band only for t <= i + KV - j0
                            if (jb == NB && (phase == 0 || i0 + rg + KV - j0 + 1 >= NB)) {
                                // a column's offset in its 16-byte superset repeats every E16 columns
                                const C *p[E16];
#pragma unroll
                                for (int x = 0; x < E16; ++x)
                                    p[x] = P + rg + lane + x * pld + (int)((o0 + x * od) & (E16 - 1));
#pragma unroll 2
                                for (int t = 0; t < NB; t += 4) {
                                    C l[4][RR];
#pragma unroll
                                    for (int x = 0; x < 4; ++x)
#pragma unroll
                                        for (int a = 0; a < RR; ++a)
                                            l[x][a] = p[x % E16][(x / E16) * E16 * pld + 32 * a];
#pragma unroll
                                    for (int x = 0; x < E16; ++x) p[x] += 4 * pld;
#pragma unroll
                                    for (int x = 0; x < 4; ++x) {
                                        C v[CG];
                                        sv_get<CG>(y + (t + x) * LC, v);
#pragma unroll
                                        for (int a = 0; a < RR; ++a)
#pragma unroll
                                            for (int c = 0; c < CG; ++c) acc[a][c] = cfms(acc[a][c], l[x][a], v[c]);
                                    }
                                }
                            } else {
#pragma unroll
                                for (int a = 0; a < RR; ++a) {
                                    const int rr = min(rg + lane + 32 * a, len - 1), i = i0 + rr;
                                    const int tm = phase ? min(jb, i + KV - j0 + 1) : jb;
                                    for (int t = 0; t < tm; ++t) {
                                        const C l = P[t * pld + (int)((o0 + t * od) & (E16 - 1)) + rr];
#pragma unroll
                                        for (int c = 0; c < CG; ++c) acc[a][c] = cfms(acc[a][c], l, y[t * LC + c]);
                                    }
                                }
                            }
                            __syncwarp();
#pragma unroll
                            for (int a = 0; a < RR; ++a)
                                if (rg + lane + 32 * a < len) sv_put<CG>(wr[a], acc[a]);
                        }
                    }
                }
                sv_arrive(SV_EMPTY + u, handover);
                if (++u == nslot) u = 0;
                ra += rc;
                if (ra >= rows) break;
                slot = slots + u * slot_bytes;
                sv_sync(SV_FULL + u, handover);
            }
            // the entering rows take the places of the block's own rows and of free ones
#pragma unroll
            for (int k = 0; k < NE; ++k) {
                const int e = tid + k * CT, c = e / NB;
                const int off = phase ? -NB - KV + e % NB : NB + kl + e % NB;
                if (c < LC) W[wrow(off) * WLD + c] = in[k];
            }
            jb0 += phase ? -NB : NB;
            if (jb0 >= WR) jb0 -= WR;
            if (jb0 < 0) jb0 += WR;
        }
        sv_sync(SV_BAR, CT);
    }
}

// ---------------------------------------------------------------------------
static int bp_grid(int64_t tasks) {
    return (int)std::max<int64_t>(1, std::min<int64_t>((tasks + BP_WARPS - 1) / BP_WARPS, 152 * 8));
}

cudaError_t launch_block_perm(int32_t *bperm, const int32_t *piv, int n, int kl, int ku, int nb, int N,
                              cudaStream_t s) {
    if (kl + nb > BP_MAXR) return cudaErrorInvalidValue;
    const int nblk = (n + nb - 1) / nb;
    block_perm_kernel<<<bp_grid((int64_t)N * nblk), BP_WARPS * 32, 0, s>>>(bperm, piv, n, kl, ku, nb, nblk, N);
    return cudaGetLastError();
}

// window rows: every row live at once and the NB that enter, rounded up to a
// multiple of the block size so that the NB rows of a block never wrap around
static int sv_window(const BandGeom &g, int nb) { return (g.kl + g.ku + 2 * nb + nb - 1) / nb * nb; }

// Bands for which the streaming solve is taken: a window without its padding
// columns and three units of 128 rows fit in shared memory, for the widest shape
// (kl + ku up to 576 in complex64, 736 in complex128, 2272 and 2352 in their real
// counterparts); wider ones take the one-kernel solve.  At the line (half-bandwidth
// 288, n = 6000, 64 points, 32 right-hand sides) a first solve takes 2.6 ms here and
// 12.4 ms there, a whole refined sampling 154 and 173 ms.  The launch needs less
// than this line asks for (sv_launch: down to two units of 32 rows).
template <typename C, int NB, int LC> static size_t sv_need(const BandGeom &g) {
    using LY = SvLayout<C, NB, LC>;
    const int WR = (g.kl + g.ku + 3 * NB + NB - 1) / NB * NB;
    return LY::smem(WR, 128, 3) - LY::w_bytes(WR) + sizeof(C) * (size_t)WR * (LC + 1);
}
size_t band_solve2_smem_c64(const BandGeom &g) { return sv_need<float2, NB_C64, 16>(g); }
size_t band_solve2_smem_c128(const BandGeom &g) { return sv_need<double2, NB_C128, 8>(g); }
size_t band_solve2_smem_r32(const BandGeom &g) { return sv_need<float, NB_C64, 16>(g); }
size_t band_solve2_smem_r64(const BandGeom &g) { return sv_need<double, NB_C128, 8>(g); }

// the shape of a refinement sweep's solve, from the number of points still
// active: the narrowest of 16, 8, 4, 2 right-hand sides per CTA whose CTAs
// for the active points fit in one wave over the SMs (a narrower shape
// shortens every block step of the chain), else the widest; gate = 0, 1, 2, 3
__global__ void solve_gate_kernel(const int32_t *__restrict__ done, int N, int L, int sms,
                                  int32_t *__restrict__ gate) {
    __shared__ int cnt;
    if (threadIdx.x == 0) cnt = 0;
    __syncthreads();
    int c = 0;
    for (int i = threadIdx.x; i < N; i += blockDim.x) c += done[i] == 0 ? 1 : 0;
    atomicAdd(&cnt, c);
    __syncthreads();
    if (threadIdx.x == 0) {
        int g = 0;
        for (int k = 3; k >= 1; --k) {
            const int lc = 16 >> k;
            if ((long long)cnt * ((L + lc - 1) / lc) <= sms) { g = k; break; }
        }
        *gate = g;
    }
}

cudaError_t launch_solve_gate(const int32_t *done, int N, int L, int sms, int32_t *gate, cudaStream_t s) {
    solve_gate_kernel<<<1, 256, 0, s>>>(done, N, L, sms, gate);
    return cudaGetLastError();
}


template <typename C, int NB, int LC, int CW, int RR, int CG>
static cudaError_t sv_launch(const C *ab, const int32_t *bperm, const C *dinv, C *B, const BandGeom &g,
                             int N, int n, int L, const int32_t *skip, const int32_t *gate, int want,
                             cudaStream_t s) {
    using LY = SvLayout<C, NB, LC>;
    const int limit = std::min(smem_optin_limit(), 227 * 1024), wr = sv_window(g, NB);
    // a unit holds a block's whole panel when there are no interchanges (at
    // most 256 rows); four slots when they fit, else two
    int rc = std::min(256, (std::max(std::max(g.kl, g.ku), 1) + 31) / 32 * 32), nslot = 4;
    if (LY::smem(wr, rc, nslot) > (size_t)limit) nslot = 2;
    while (rc > 32 && LY::smem(wr, rc, nslot) > (size_t)limit) rc -= 32;
    const size_t smem = LY::smem(wr, rc, nslot);
    if (smem > (size_t)limit) return cudaErrorInvalidConfiguration;
    cudaError_t e = cudaFuncSetAttribute(band_solve_stream_kernel<C, NB, LC, CW, RR, CG>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, limit);
    if (e != cudaSuccess) return e;
    dim3 grid((L + LC - 1) / LC, N);
    band_solve_stream_kernel<C, NB, LC, CW, RR, CG><<<grid, 32 * CW + SV_PRODUCERS, smem, s>>>(
        ab, bperm, dinv, B, n, g.kl, g.ku, g.ldab, L, wr, rc, nslot, skip, gate, want);
    return cudaGetLastError();
}

// Computing warps (CW) and the rows (RR) and columns (CG) a lane updates.
// Shared memory returns 128 bytes a cycle to the lanes, broadcasts included, so
// one row by eight columns a lane (sixteen warps) was bound by its loads: 7500
// cycles a step at half-bandwidth 200 with 16 right-hand sides, 3600 of FMAs;
// four rows by four columns on eight warps need as many cycles of loads as of
// FMAs.  With fewer right-hand sides, and for narrow bands, a step is a chain of
// latencies and a warp alone issues an instruction every three cycles: there
// sixteen warps with small tasks are faster than four with large ones (2-column
// sweeps 5.5 against 6.9 ms).
template <typename C, int NB, int LC>
static cudaError_t sv_dispatch(const C *ab, const int32_t *bperm, const C *dinv, C *B, const BandGeom &g, int N,
                               int n, int L, const int32_t *skip, const int32_t *gate, int want, cudaStream_t s) {
    const int groups = (std::min(256, std::max(g.kl, g.ku)) + 31) / 32;  // of 32 rows
#define SV_GO(CW, RR, CG) return sv_launch<C, NB, LC, CW, RR, CG>(ab, bperm, dinv, B, g, N, n, L, skip, gate, want, s)
    if constexpr (sizeof(typename real_of<C>::type) == 8) {
        SV_GO(16, 1, 1);
    } else if constexpr (LC == 16) {
        if (groups >= 5) SV_GO(8, 4, 4);
        if (groups >= 3) SV_GO(8, 2, 4);
        SV_GO(16, 1, 2);
    } else if constexpr (LC == 8) {
        if (groups >= 5) SV_GO(16, 1, 4);
        if (groups >= 3) SV_GO(16, 1, 2);
        SV_GO(16, 1, 1);
    } else if constexpr (LC == 4) {
        if (groups >= 5) SV_GO(16, 1, 2);
        SV_GO(16, 1, 1);
    } else {
        SV_GO(16, 1, 1);
    }
#undef SV_GO
}

// right-hand sides per CTA when the caller leaves it open (0): the narrowest
// shape whose CTAs fit the SMs at once (a narrower one shortens every step of
// the chain), else the widest
template <int WIDEST> static int sv_columns(int N, int L) {
    int dev = 0, sms = 152;
    if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    for (int lc = 2; lc < WIDEST; lc *= 2)
        if ((int64_t)N * ((L + lc - 1) / lc) <= sms) return lc;
    return WIDEST;
}

cudaError_t launch_band_solve2_c64(const float2 *ab, const int32_t *bperm, const float2 *dinv,
                                   float2 *B, const BandGeom &g, int N, int n, int L,
                                   const int32_t *skip, cudaStream_t s, int lc,
                                   const int32_t *gate, int want) {
    switch (lc ? lc : sv_columns<16>(N, L)) {
    case 2: return sv_dispatch<float2, NB_C64, 2>(ab, bperm, dinv, B, g, N, n, L, skip, gate, want, s);
    case 4: return sv_dispatch<float2, NB_C64, 4>(ab, bperm, dinv, B, g, N, n, L, skip, gate, want, s);
    case 8: return sv_dispatch<float2, NB_C64, 8>(ab, bperm, dinv, B, g, N, n, L, skip, gate, want, s);
    default: return sv_dispatch<float2, NB_C64, 16>(ab, bperm, dinv, B, g, N, n, L, skip, gate, want, s);
    }
}
cudaError_t launch_band_solve2_r32(const float *ab, const int32_t *bperm, const float *dinv, float *B,
                                   const BandGeom &g, int N, int n, int L, const int32_t *skip, cudaStream_t s) {
    switch (sv_columns<16>(N, L)) {
    case 2:
    case 4: return sv_dispatch<float, NB_C64, 4>(ab, bperm, dinv, B, g, N, n, L, skip, nullptr, 0, s);
    default: return sv_dispatch<float, NB_C64, 16>(ab, bperm, dinv, B, g, N, n, L, skip, nullptr, 0, s);
    }
}
template <typename C>
static cudaError_t sv_double(const C *ab, const int32_t *bperm, const C *dinv, C *B, const BandGeom &g, int N, int n,
                             int L, const int32_t *skip, cudaStream_t s) {
    switch (sv_columns<8>(N, L)) {
    case 2: return sv_dispatch<C, NB_C128, 2>(ab, bperm, dinv, B, g, N, n, L, skip, nullptr, 0, s);
    case 4: return sv_dispatch<C, NB_C128, 4>(ab, bperm, dinv, B, g, N, n, L, skip, nullptr, 0, s);
    default: return sv_dispatch<C, NB_C128, 8>(ab, bperm, dinv, B, g, N, n, L, skip, nullptr, 0, s);
    }
}
cudaError_t launch_band_solve2_r64(const double *ab, const int32_t *bperm, const double *dinv, double *B,
                                   const BandGeom &g, int N, int n, int L, const int32_t *skip, cudaStream_t s) {
    return sv_double(ab, bperm, dinv, B, g, N, n, L, skip, s);
}
cudaError_t launch_band_solve2_c128(const double2 *ab, const int32_t *bperm, const double2 *dinv,
                                    double2 *B, const BandGeom &g, int N, int n, int L,
                                    const int32_t *skip, cudaStream_t s) {
    return sv_double(ab, bperm, dinv, B, g, N, n, L, skip, s);
}

}  // namespace rsrr
