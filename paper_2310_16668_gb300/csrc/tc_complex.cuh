// Tensor-core translations for the complex 3D Helmholtz kernel (FP32_TC,
// complex64): the building blocks of tc_kernels.cuh (bulk-copy stages,
// mbarrier protocol with bounded waits, TMEM accumulators, 3-pass TF32 split)
// applied to e^{i kappa r} / (4 pi r), with the sine and cosine evaluated on
// the FP32 pipe.
#pragma once

#include "tc_kernels.cuh"

namespace skel {

// ---------------------------------------------------------------------------
// 3D Helmholtz (complex64) on the tensor cores: u = G q with G = G_r + i G_i
// and q = q_r + i q_i is u_r = G_r q_r - G_i q_i, u_i = G_r q_i + G_i q_r, so
// one real accumulator of 32 columns holds [u_r | u_i] of 16 right-hand sides
// as G_r B + G_i B' with B = [q_r | q_i] and B' = [-q_i | q_r]
// (tc_bprep_kernel<true> writes both, TF32 hi + lo).
//
// As in the real kernel (tc_near.cuh) the hi*hi products of a pair of tiles
// accumulate in D, the small products in L, and hi * [hi | lo] is one MMA into
// both: 16 MMAs a tile. Pairs alternate between two (D, L); the pair before
// last is added to the register sums when a pair starts. Tensor memory: two
// (D, L) (128 columns) and three A buffers of G_r hi, G_r lo, G_i hi, G_i lo
// (3 x 128): 512 columns, one CTA per SM, so the CTA brings its own latency
// hiding: 4 compute threads per row (16 compute warps), 8 sources of a tile
// each. Masks as in tc_near.cuh.
// Bound by the FP32 pipe: about 60 paired instructions for two values with
// their split; the MMAs take 16 x 48 of a tile's cycles. FP32, kappa 25, 16
// right-hand sides, leaves of 128, before (24 MMAs, quadrant selection, a copy
// of the coordinates per slot) and after: N = 20,011 602 -> 531 us, 4,000
// 152 -> 138, 1,000 (5 right-hand sides) 60 -> 52; error against complex128
// 8.4e-7 -> 7.4e-7.
constexpr int kTcNc = 16;                      // complex right-hand sides per pass
constexpr uint32_t kTmemColsC = 512;
constexpr uint32_t kColAc = 128;               // A[b]: G_r hi, G_r lo, G_i hi, G_i lo at 128 + 128 b (+0/32/64/96)
constexpr int kChunkFloatsC = 4 * 1024 + 2 * 96;
constexpr int kTprC = 4;                       // compute threads per target row
constexpr int kComputeC = 128 * kTprC;         // compute threads
constexpr int kSrcC = 32 / kTprC;              // sources of a tile per compute thread
constexpr int kColsC = kTcN / kTprC;           // accumulator columns per compute thread
constexpr int kThreadsC = kComputeC + 64;      // + the producer warp and the MMA warp
struct alignas(128) TcStageC {
    float b[2 * 1024];                         // B = [q_r | q_i], TF32 hi and lo
    float bp[2 * 1024];                        // B' = [-q_i | q_r], TF32 hi and lo
    float xh[3 * 32];                          // source coordinates (hi): x, y, z
    float xl[3 * 32];                          // lo parts (touching-leaf tiles)
    SrcTile tile;                              // the tile's descriptor (its own copy)
};
static_assert(offsetof(TcStageC, tile) == kChunkFloatsC * 4, "chunk blob is contiguous in the stage");
constexpr int kNSC = 6;                        // data stages
template <int NS>
struct TcSharedC {
    TcStageC st[NS];
    float outer[kColsC][kComputeC];
    uint64_t full[NS], afull[NS], empty[NS];
    uint32_t tmem;
};
constexpr int kTccSmemRequest = 144 * 1024;   // one CTA per SM (512 TMEM columns)
static_assert(sizeof(TcSharedC<kNSC>) <= kTccSmemRequest, "shared memory plan");

__device__ __forceinline__ float2 tc_f2(float x) { return make_float2(x, x); }

__device__ __forceinline__ void tmem_ld8(uint32_t taddr, uint32_t* v) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7])
                 : "r"(taddr) : "memory");
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

// (-1)^n sin x and (-1)^n cos x of two non-negative arguments x up to 2^21,
// with n = x / pi rounded to nearest, whose parity comes back in bit 0 of nx
// and ny: x = n pi + y with |y| <= pi/2. n is rounded by adding 1.5 * 2^23 (the
// sum's low mantissa bits are then n: no conversion instruction); Cody and
// Waite's reduction with pi as a sum of three floats, the first with 9
// significant bits so that n C1 is exact; the Taylor series of sin y to the
// y^13 term (truncation below 7e-10 on |y| <= pi/2) and of cos y to the y^14
// term (below 7e-11). Reducing by pi instead of pi/2 takes three more
// coefficients but no choice between the two series and one sign for both,
// which the caller puts on the common factor 1/r: two integer instructions a
// value instead of ten. FP32 pipe only, two arguments per paired instruction.
__device__ __forceinline__ void tc_sincos2(float2 x, float2& s, float2& c, uint32_t& nx, uint32_t& ny) {
    constexpr double kPi = 3.14159265358979323846264338327950;
    constexpr float kC1 = 3.140625f;
    constexpr float kC2 = (float)(kPi - 3.140625);
    constexpr float kC3 = (float)(kPi - 3.140625 - (double)kC2);
    constexpr float kRound = 12582912.0f;      // 1.5 * 2^23
    const float2 t = __ffma2_rn(x, tc_f2((float)(1.0 / kPi)), tc_f2(kRound));
    const float2 mn = __ffma2_rn(t, tc_f2(-1.f), tc_f2(kRound));   // -n (exact)
    float2 y = __ffma2_rn(mn, tc_f2(kC1), x);
    y = __ffma2_rn(mn, tc_f2(kC2), y);
    y = __ffma2_rn(mn, tc_f2(kC3), y);
    const float2 z = __fmul2_rn(y, y);
    float2 ps = __ffma2_rn(z, tc_f2((float)(1.0 / 6227020800.0)), tc_f2((float)(-1.0 / 39916800.0)));
    ps = __ffma2_rn(z, ps, tc_f2((float)(1.0 / 362880.0)));
    ps = __ffma2_rn(z, ps, tc_f2((float)(-1.0 / 5040.0)));
    ps = __ffma2_rn(z, ps, tc_f2((float)(1.0 / 120.0)));
    ps = __ffma2_rn(z, ps, tc_f2((float)(-1.0 / 6.0)));
    s = __ffma2_rn(__fmul2_rn(y, z), ps, y);
    float2 pc = __ffma2_rn(z, tc_f2((float)(-1.0 / 87178291200.0)), tc_f2((float)(1.0 / 479001600.0)));
    pc = __ffma2_rn(z, pc, tc_f2((float)(-1.0 / 3628800.0)));
    pc = __ffma2_rn(z, pc, tc_f2((float)(1.0 / 40320.0)));
    pc = __ffma2_rn(z, pc, tc_f2((float)(-1.0 / 720.0)));
    pc = __ffma2_rn(z, pc, tc_f2((float)(1.0 / 24.0)));
    pc = __ffma2_rn(z, pc, tc_f2(-0.5f));
    c = __ffma2_rn(z, pc, tc_f2(1.0f));
    nx = __float_as_uint(t.x);
    ny = __float_as_uint(t.y);
    asm volatile("" : "+r"(nx), "+r"(ny));     // (as in tc_log8)
}

// e^{i kappa r} / r without its 1/(4 pi) for 8 sources (coordinates at x: 32
// floats per axis, lo parts 96 floats on), split into TF32 hi and lo: the
// reciprocal square root as in the real path (0 at kFar and, on touching
// leaves, for r^2 <= FLT_MIN), r = r^2 / r corrected by one Newton step, then
// tc_sincos2 of kappa r. A zero reciprocal makes r a NaN or 0; the minimum
// with 2^21 turns that (and only that: kappa r stays far below) into a finite
// argument, whose sine and cosine the zero reciprocal then cancels.
// kb: the row's kept sources (bit per source), used if CUT.
template <bool ADJ, bool CUT>
__device__ __forceinline__ void tc_ceval(const float* x, float4 nt, float4 nl, float kappa, uint32_t kb, uint32_t* grh,
                                         uint32_t* grl, uint32_t* gih, uint32_t* gil) {
    constexpr int AX = 32, LO = 96;
    const float2 ntx = tc_f2(nt.x), nty = tc_f2(nt.y), ntz = tc_f2(nt.z);
    const float2 m1 = tc_f2(-1.f), split = tc_f2(8193.f), kap = tc_f2(kappa);
#pragma unroll
    for (int q = 0; q < kSrcC / 4; ++q) {
        const float4 X = *reinterpret_cast<const float4*>(x + 4 * q);
        const float4 Y = *reinterpret_cast<const float4*>(x + AX + 4 * q);
        const float4 Z = *reinterpret_cast<const float4*>(x + 2 * AX + 4 * q);
        float4 LX, LY, LZ;
        if (ADJ) {
            LX = *reinterpret_cast<const float4*>(x + LO + 4 * q);
            LY = *reinterpret_cast<const float4*>(x + LO + AX + 4 * q);
            LZ = *reinterpret_cast<const float4*>(x + LO + 2 * AX + 4 * q);
        }
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int jj = 4 * q + 2 * h;
            float2 dx = __fadd2_rn(h ? make_float2(X.z, X.w) : make_float2(X.x, X.y), ntx);
            float2 dy = __fadd2_rn(h ? make_float2(Y.z, Y.w) : make_float2(Y.x, Y.y), nty);
            float2 dz = __fadd2_rn(h ? make_float2(Z.z, Z.w) : make_float2(Z.x, Z.y), ntz);
            if (ADJ) {
                dx = __fadd2_rn(dx, __fadd2_rn(h ? make_float2(LX.z, LX.w) : make_float2(LX.x, LX.y), tc_f2(nl.x)));
                dy = __fadd2_rn(dy, __fadd2_rn(h ? make_float2(LY.z, LY.w) : make_float2(LY.x, LY.y), tc_f2(nl.y)));
                dz = __fadd2_rn(dz, __fadd2_rn(h ? make_float2(LZ.z, LZ.w) : make_float2(LZ.x, LZ.y), tc_f2(nl.z)));
            }
            float2 r2 = __fmul2_rn(dx, dx);
            r2 = __ffma2_rn(dy, dy, r2);
            r2 = __ffma2_rn(dz, dz, r2);
            float2 ri = make_float2(tc_rsqrt<ADJ>(r2.x), tc_rsqrt<ADJ>(r2.y));
            float2 r = __fmul2_rn(r2, ri);
            r = __ffma2_rn(r, __ffma2_rn(r, __fmul2_rn(ri, tc_f2(-0.5f)), tc_f2(0.5f)), r);
            float2 kr = __fmul2_rn(kap, r);
            kr.x = fminf(kr.x, 2097152.f);
            kr.y = fminf(kr.y, 2097152.f);
            if (CUT) {
                ri.x = (kb >> jj) & 1u ? ri.x : 0.f;
                ri.y = (kb >> (jj + 1)) & 1u ? ri.y : 0.f;
            }
            float2 sn, cs;
            uint32_t nx, ny;
            tc_sincos2(kr, sn, cs, nx, ny);
            ri.x = __uint_as_float(__float_as_uint(ri.x) ^ (nx << 31));
            ri.y = __uint_as_float(__float_as_uint(ri.y) ^ (ny << 31));
            const float2 gR = __fmul2_rn(cs, ri), gI = __fmul2_rn(sn, ri);
            // Veltkamp's split of both parts (as tc_split_store)
            const float2 tR = __fmul2_rn(gR, split), tI = __fmul2_rn(gI, split);
            const float2 hR = __ffma2_rn(__ffma2_rn(gR, m1, tR), m1, tR);
            const float2 hI = __ffma2_rn(__ffma2_rn(gI, m1, tI), m1, tI);
            const float2 lR = __ffma2_rn(hR, m1, gR), lI = __ffma2_rn(hI, m1, gI);
            grh[jj] = __float_as_uint(hR.x), grh[jj + 1] = __float_as_uint(hR.y);
            grl[jj] = __float_as_uint(lR.x), grl[jj + 1] = __float_as_uint(lR.y);
            gih[jj] = __float_as_uint(hI.x), gih[jj + 1] = __float_as_uint(hI.y);
            gil[jj] = __float_as_uint(lI.x), gil[jj + 1] = __float_as_uint(lI.y);
        }
    }
}

// One CTA per tensor-core item, the roles and barriers of tc_near_kernel
// (kComputeC compute threads); 16 complex right-hand sides per pass
// (a.r0 .. a.r0 + 15), U complex64 rows.
template <int NS = kNSC>
__global__ void __launch_bounds__(kThreadsC, 1) tc_cnear_kernel(const TcArgs a) {
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    TcSharedC<NS>& S = *reinterpret_cast<TcSharedC<NS>*>(smem_raw);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const TcItem* itp = a.items + blockIdx.x;
    const int64_t row_off = itp->row_off;
    const int nrows = itp->nrows, nslot = itp->nslot, list_lo = itp->list_lo;
    const int ntile = itp->list_hi - list_lo;

    if (tid == 0) {
        for (int s = 0; s < NS; ++s) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" :: "r"(sm_addr(&S.full[s])));
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" :: "r"(sm_addr(&S.afull[s])), "r"(kComputeC));
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" :: "r"(sm_addr(&S.empty[s])));
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     :: "r"(sm_addr(&S.tmem)), "r"(kTmemColsC));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tbase = S.tmem;
    bool err = false;

    if (warp == kComputeC / 32) {
        // ---------------- producer warp ----------------
        for (int t0 = 0; t0 < ntile; t0 += 32) {
            const int d_chunk = t0 + lane < ntile ? a.tiles[list_lo + t0 + lane].chunk : 0;
            const int nb = min(32, ntile - t0);
            for (int i = 0; i < nb; ++i) {
                const int t = t0 + i;
                const int s = t % NS;
                const int chunk = __shfl_sync(0xffffffffu, d_chunk, i);
                if (t >= NS && !mbar_wait(sm_addr(&S.empty[s]), (uint32_t)(((t - NS) / NS) & 1), a.wait_ns)) err = true;
                const bool hold = t == 0 && (int)blockIdx.x == a.withhold_item;
                if (hold && !withhold_first_tile(sm_addr(&S.afull[0]), a.wait_ns)) err = true;
                if (lane == 0) {
                    const uint32_t bar = sm_addr(&S.full[s]);
                    mbar_arrive_tx(bar, 4u * kChunkFloatsC + 64u);
                    bulk_g2s_hint(sm_addr(S.st[s].b), a.B + (int64_t)chunk * kChunkFloatsC, 4u * kChunkFloatsC, bar,
                                  l2_evict_last());
                    bulk_g2s_hint(sm_addr(&S.st[s].tile), a.tiles + list_lo + t, 64u, bar, l2_evict_first());
                    if (hold && !mbar_wait(bar, 0u, a.wait_ns)) err = true;
                }
                __syncwarp();
            }
        }
        if (lane == 0) {
            for (int t = (ntile > NS ? ntile - NS : 0); t < ntile; ++t)
                if (!mbar_wait(sm_addr(&S.full[t % NS]), (uint32_t)((t / NS) & 1), a.wait_ns)) err = true;
        }
    } else if (warp == kComputeC / 32 + 1) {
        // ---------------- MMA issuer (one thread) ----------------
        if (lane == 0) {
            const uint32_t idesc32 =
                (1u << 4) | (2u << 7) | (2u << 10) | ((uint32_t)(kTcN >> 3) << 17) | ((128u >> 4) << 24);
            const uint32_t idesc64 =
                (1u << 4) | (2u << 7) | (2u << 10) | ((uint32_t)(2 * kTcN >> 3) << 17) | ((128u >> 4) << 24);
            for (int m = 0; m < ntile; ++m) {
                const int s = m % NS, ab = m % kNA;
                if (!mbar_wait(sm_addr(&S.afull[s]), (uint32_t)((m / NS) & 1), a.wait_ns)) err = true;
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                const uint32_t b0 = smem_desc_lo(sm_addr(S.st[s].b)), bp0 = smem_desc_lo(sm_addr(S.st[s].bp));
                const uint32_t d = tbase + 64u * ((uint32_t)(m >> 1) & 1u), l = d + 32u;
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const uint32_t ar = tbase + kColAc + 128u * ab + 8u * k, ai = ar + 64u;
                    const uint32_t db = b0 + kDescStep * k, dbp = bp0 + kDescStep * k;
                    mma_tf32_lo(d, ar, db, idesc64, true);             // D, L += G_r hi [hi | lo]
                    mma_tf32_lo(l, ar + 32u, db, idesc32, true);       // L += G_r lo hi
                    mma_tf32_lo(d, ai, dbp, idesc64, true);
                    mma_tf32_lo(l, ai + 32u, dbp, idesc32, true);
                }
                asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];"
                             :: "r"(sm_addr(&S.empty[s])) : "memory");
            }
        }
    } else {
        // ---------------- compute warps: thread (row, quarter) ----------------
        const int row = tid & 127, quarter = tid >> 7;
        const bool valid = row < nrows;
        int myslot = 0;
        for (int c = 1; c < nslot; ++c)
            if (row >= itp->slot_start[c]) myslot = c;
        float4 tx = make_float4(0.f, 0.f, 0.f, 0.f), tl = tx;
        if (valid) {
            tx = a.X[row_off + row];
            tl = a.Xlo[row_off + row];
        }
        const uint32_t lane_off = (uint32_t)((warp & 3) * 32) << 16;
        const int j0 = kSrcC * quarter;
        const uint32_t dcol = tbase + lane_off + (uint32_t)(kColsC * quarter);
        float acc[kColsC];
#pragma unroll
        for (int c = 0; c < kColsC; ++c) {
            acc[c] = 0.f;
            S.outer[c][tid] = 0.f;
        }
        const uint32_t zero[8] = {0u, 0u, 0u, 0u, 0u, 0u, 0u, 0u};
        auto clear = [&]() {                                   // this thread's columns of both (D, L)
#pragma unroll
            for (int i = 0; i < 4; ++i) tmem_st8(dcol + 32u * i, zero);
        };
        auto add = [&](uint32_t taddr) {
            uint32_t v[kColsC];
            tmem_ld8(taddr, v);
#pragma unroll
            for (int c = 0; c < kColsC; ++c) acc[c] += __uint_as_float(v[c]);
        };
        // tile m's MMAs are done: asked for early, settled when it matters
        auto ask = [&](int m) { return mbar_test(sm_addr(&S.empty[m % NS]), (uint32_t)((m / NS) & 1)); };
        auto settle = [&](uint32_t early, int m) {
            if (!mbar_settle(early, sm_addr(&S.empty[m % NS]), (uint32_t)((m / NS) & 1), a.wait_ns)) err = true;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        };
        // everything accumulated in tensor memory before tile u of the group
        // that starts at s0, to the outer sums
        auto flush = [&](int u, int s0) {
            if (u <= s0) return;
            settle(ask(u - 1), u - 1);
            const int np = (u - s0 + 1) / 2;
            for (int p = max(np - 2, 0); p < np; ++p) add(dcol + 64u * ((uint32_t)p & 1u));
            add(dcol + 32u);
            add(dcol + 96u);
#pragma unroll
            for (int c = 0; c < kColsC; ++c) {
                S.outer[c][tid] += acc[c];
                acc[c] = 0.f;
            }
        };
        clear();
        uint32_t landed = 0u;                                  // the next tile's copies, asked for early
        for (int u = 0; u < ntile; ++u) {
            const int s = u % NS;
            if (!mbar_settle(landed, sm_addr(&S.full[s]), (uint32_t)((u / NS) & 1), a.wait_ns)) err = true;
            landed = mbar_test(sm_addr(&S.full[(u + 1) % NS]), (uint32_t)(((u + 1) / NS) & 1));
            const uint32_t early = u >= 3 ? ask(u - 3) : 0u;
            const TcStageC& st = S.st[s];
            const bool adj = (st.tile.flags & TASK_ADJ) != 0;
            const uint32_t all = st.tile.cnt >= 32 ? 0xFFFFFFFFu : (1u << (st.tile.cnt & 31)) - 1u;
            float4 nt, nl;
            tc_frame(tx, tl, st.tile.cen, adj, nt, nl);
            const uint32_t kb = valid ? (st.tile.keep[myslot] >> j0) & 0xFFu : 0u;
            const bool none = __all_sync(0xffffffffu, kb == 0u);
            const bool cut = __any_sync(0xffffffffu, kb != 0u && kb != (all >> j0 & 0xFFu));
            if (kb == 0u) nt.x = kFar;                         // the row keeps none of these sources
            uint32_t grh[kSrcC], grl[kSrcC], gih[kSrcC], gil[kSrcC];
            if (none) {
#pragma unroll
                for (int jj = 0; jj < kSrcC; ++jj) grh[jj] = grl[jj] = gih[jj] = gil[jj] = 0u;
            } else if (adj) {
                if (cut) tc_ceval<true, true>(st.xh + j0, nt, nl, a.kappa, kb, grh, grl, gih, gil);
                else tc_ceval<true, false>(st.xh + j0, nt, nl, a.kappa, kb, grh, grl, gih, gil);
            } else {
                if (cut) tc_ceval<false, true>(st.xh + j0, nt, nl, a.kappa, kb, grh, grl, gih, gil);
                else tc_ceval<false, false>(st.xh + j0, nt, nl, a.kappa, kb, grh, grl, gih, gil);
            }
            __syncwarp();
            const int g = u & (kTcOuter - 1);                  // tile of the group
            if (u > 0 && g == 0) {
                flush(u, u - kTcOuter);
                clear();
            } else if (u >= 3) {
                // A buffer u % 3 was last read by MMA(u - 3)
                settle(early, u - 3);
                // the pair two before the one that starts here, which restarts its D
                if (g >= 4 && !(g & 1)) {
                    const uint32_t dc = dcol + 64u * ((uint32_t)(g >> 1) & 1u);
                    add(dc);
                    tmem_st8(dc, zero);
                }
            }
            const uint32_t acol = tbase + lane_off + kColAc + 128u * (u % kNA) + (uint32_t)j0;
            tmem_st8(acol, grh);
            tmem_st8(acol + 32u, grl);
            tmem_st8(acol + 64u, gih);
            tmem_st8(acol + 96u, gil);
            asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            mbar_arrive(sm_addr(&S.afull[s]));
        }
        flush(ntile, ntile > 0 ? (ntile - 1) & ~(kTcOuter - 1) : 0);
#pragma unroll
        for (int c = 0; c < kColsC; ++c) acc[c] = S.outer[c][tid];
        if (valid) {
            // quarter q holds columns 8q .. 8q + 7: real parts of right-hand
            // sides r0 + 8 (q & 1) .. + 7 (q < 2), their imaginary parts (q >= 2)
            const float scale = (float)green_scale<2>();
            const int64_t base = (row_off + row) * a.nrhs;
            const int c0 = a.r0 + kColsC * (quarter & 1), part = quarter >> 1;
#pragma unroll
            for (int c = 0; c < kColsC; ++c)
                if (c0 + c < a.nrhs) a.U[2 * (base + c0 + c) + part] = scale * acc[c];
        }
    }
    if (err) atomicExch(a.status, 1);
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 0) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" :: "r"(tbase), "r"(kTmemColsC));
    }
}

}  // namespace skel
