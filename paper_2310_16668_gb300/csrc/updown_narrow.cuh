// Upward / downward passes for few right-hand sides (nrhs <= 8): the skeleton
// GEMMs are then matrix-vector products, bound by reading T once. The kernels
// of skel_kernels.cuh and updown_async.cuh put a right-hand side on every lane
// (31 of 32 lanes idle at nrhs = 1, and FP64 multiply-adds cost the same for
// idle lanes); here a lane owns an output row.
//
// A work-list entry is 32 output rows of one box. Its inner index is cut into
// at most 8 segments (un_segment() long, from the box alone), whose partial
// sums are added in order. W = 8: a CTA of 8 warps per entry, one per segment;
// W = 1: 8 entries per CTA, each warp runs through its entry's segments, for
// levels whose boxes have at most two (2D trees: 64 curve sets at 4 columns
// took 0.19 ms a pass with a CTA per entry). Per inner index a warp loads one
// coalesced column of 32 T entries (16 in flight) and the row's RT values from
// a staged block. Every shape gives the same bits.
// 64 curve sets, 4 right-hand sides, up + down per apply: 246 -> 209 us.
#pragma once

#include "skel_kernels.cuh"

namespace skel {

constexpr int kUnWarps = 8;                // warps per CTA; segments of an entry, at most
constexpr int kUnMaxRhs = 8;
__host__ __device__ constexpr int un_segment(int ninner) {
    const int eighth = ((ninner + 7) / 8 + 31) / 32 * 32;
    return eighth > 64 ? eighth : 64;
}

template <class S, bool DOWN, int RT, int W>
__global__ void __launch_bounds__(32 * kUnWarps) updown_narrow_kernel(const UpBox* __restrict__ up,
                                                                      const int2* __restrict__ work, int n_work,
                                                                      const int32_t* __restrict__ pos,
                                                                      const S* __restrict__ T, S* X, int nrhs,
                                                                      bool conj_op) {
    __shared__ S sq[kUnWarps][32][RT];
    __shared__ S ps[W > 1 ? kUnWarps : 1][RT][32];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int entry = W > 1 ? (int)blockIdx.x : (int)blockIdx.x * kUnWarps + warp;
    if (entry >= n_work) return;
    const int2 w = work[entry];
    const UpBox u = up[w.x];
    const int k = u.k, r = u.n - u.k;
    const int nout = DOWN ? r : k, ninner = DOWN ? k : r;
    const int row0 = w.y;
    const int tid = W > 1 ? (int)threadIdx.x : lane;         // thread of the entry, of 32 W
    if (DOWN && row0 == 0) {                                 // u_S += uhat
        for (int i = tid; i < k * nrhs; i += 32 * W) {
            const int e = i / nrhs, c = i - e * nrhs;
            const int64_t at = (u.off + pos[u.off + e]) * nrhs + c;
            X[at] = X[at] + X[(u.dst + e) * nrhs + c];
        }
    }
    if (row0 >= nout) return;
    const bool rowok = row0 + lane < nout;
    const int seg = un_segment(ninner), nseg = (ninner + seg - 1) / seg;
    const S* Tr = T + u.T_off + row0 + lane;
    S acc[RT], tot[RT];
#pragma unroll
    for (int c = 0; c < RT; ++c) acc[c] = tot[c] = zero<S>();
    for (int sg = W > 1 ? warp : 0; sg < nseg; sg += W) {
        const int j_hi = min((sg + 1) * seg, ninner);
        for (int j0 = sg * seg; j0 < j_hi; j0 += 32) {
            const int jn = min(32, j_hi - j0);
            if (lane < jn) {
                const int64_t e = DOWN ? u.dst + j0 + lane : u.off + pos[u.off + k + j0 + lane];
#pragma unroll
                for (int c = 0; c < RT; ++c) sq[warp][lane][c] = c < nrhs ? X[e * nrhs + c] : zero<S>();
            }
            __syncwarp();
            constexpr int G = 16;
            for (int g0 = 0; g0 < jn; g0 += G) {
                S a[G];
#pragma unroll
                for (int q = 0; q < G; ++q)
                    a[q] = rowok && g0 + q < jn ? Tr[(int64_t)(j0 + g0 + q) * nout] : zero<S>();
#pragma unroll
                for (int q = 0; q < G; ++q)
                    if (g0 + q < jn) {
                        const S v = conj_op ? conj(a[q]) : a[q];
#pragma unroll
                        for (int c = 0; c < RT; ++c) acc[c] += v * sq[warp][g0 + q][c];
                    }
            }
            __syncwarp();
        }
        if constexpr (W == 1) {
#pragma unroll
            for (int c = 0; c < RT; ++c) {
                tot[c] = sg == 0 ? acc[c] : tot[c] + acc[c];
                acc[c] = zero<S>();
            }
        }
    }
    auto row_at = [&](int orow) { return (u.off + pos[u.off + (DOWN ? k : 0) + orow]) * nrhs; };
    if constexpr (W == 1) {
        if (!rowok) return;
        const int64_t src = row_at(row0 + lane), dst = DOWN ? src : (u.dst + row0 + lane) * nrhs;
#pragma unroll
        for (int c = 0; c < RT; ++c)
            if (c < nrhs) X[dst + c] = X[src + c] + tot[c];
    } else {
#pragma unroll
        for (int c = 0; c < RT; ++c) ps[warp][c][lane] = acc[c];
        __syncthreads();
        for (int i = threadIdx.x; i < 32 * nrhs; i += 32 * W) {
            const int row = i / nrhs, c = i - row * nrhs, orow = row0 + row;
            if (orow >= nout) continue;
            S v = nseg > 0 ? ps[0][c][row] : zero<S>();
            for (int q = 1; q < nseg; ++q) v = v + ps[q][c][row];
            const int64_t src = row_at(orow) + c, dst = DOWN ? src : (u.dst + orow) * nrhs + c;
            X[dst] = X[src] + v;
        }
    }
}

}  // namespace skel
