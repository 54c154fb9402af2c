// Upward / downward passes for few right-hand sides (nrhs <= 8): the skeleton
// GEMMs are then matrix-vector products, bound by reading T once. The kernels
// of skel_kernels.cuh and updown_async.cuh put a right-hand side on every lane
// (31 of 32 lanes idle at nrhs = 1, and FP64 multiply-adds cost the same for
// idle lanes); here a lane owns an output row.
//
// A work-list entry is 32 output rows of one box. As in those kernels the inner
// index runs in chunks of 32, chunk ch in stream ch % 8 (for FP32 these are
// their streams, and the bits are theirs: one more launch shape), and the
// streams' sums are added in order. W = 8: a CTA of 8 warps per entry, a stream
// per warp; W = 1: 8 entries per CTA, each warp runs through its entry's streams.
// Per inner index a warp loads one coalesced column of 32 T entries and the row's
// RT values from a staged block; the next group of T entries, the next chunk's
// values and the entries after those are in flight while a group is multiplied.
// Latency-bound on small levels (about 6 us a launch), by the loads of T on large
// ones. FP32, 1 and 4 right-hand sides, the best column-per-lane shape against
// this kernel: 64 boxes of 174 x 797, up 42, 42 -> 12, 15 us, down 29, 26 -> 14, 17;
// 4,096 boxes of 21 x 47, up 27, 20 -> 11, 14, down 28, 26 -> 10, 15. Whole applies:
// 3D N = 65,536, one column, 595 -> 504 us; 2D N = 200,000, 4 columns, 845 -> 641;
// sphere + cluster N = 22,894, 4 columns, tuned, 217 -> 171.
#pragma once

#include "skel_kernels.cuh"

namespace skel {

constexpr int kUnWarps = 8;                // warps per CTA; streams of an entry
constexpr int kUnMaxRhs = 8;

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
    const int nch = (ninner + 31) / 32, nst = nch < kUnWarps ? nch : kUnWarps;
    const S* Tr = T + u.T_off + row0 + lane;
    constexpr int G = sizeof(S) <= 4 ? 16 : sizeof(S) <= 8 ? 8 : 4;   // T entries of a group
    // inner indices j0 .. j0 + G - 1 of this lane's row
    auto load_t = [&](int j0, S* a) {
#pragma unroll
        for (int q = 0; q < G; ++q) a[q] = rowok && j0 + q < ninner ? Tr[(int64_t)(j0 + q) * nout] : zero<S>();
    };
    // this lane's inner index of chunk ch: its entry, and its values
    auto entry_of = [&](int ch) -> int64_t {
        const int j = 32 * ch + lane;
        if (j >= ninner) return -1;
        return DOWN ? u.dst + j : u.off + pos[u.off + k + j];
    };
    auto load_x = [&](int64_t e, S* x) {
#pragma unroll
        for (int c = 0; c < RT; ++c) x[c] = e >= 0 && c < nrhs ? X[e * nrhs + c] : zero<S>();
    };
    S acc[RT], tot[RT], x[RT], a[G], b[G];
#pragma unroll
    for (int c = 0; c < RT; ++c) acc[c] = tot[c] = zero<S>();
    for (int st = W > 1 ? warp : 0; st < nst; st += W) {
        load_t(32 * st, a);
        load_x(entry_of(st), x);
        int64_t next = entry_of(st + kUnWarps);
        for (int ch = st; ch < nch; ch += kUnWarps) {
            const int jn = min(32, ninner - 32 * ch);
#pragma unroll
            for (int c = 0; c < RT; ++c) sq[warp][lane][c] = x[c];
            __syncwarp();
            load_x(next, x);
            next = entry_of(ch + 2 * kUnWarps);
#pragma unroll
            for (int g0 = 0; g0 < 32; g0 += G) {
                if (g0 >= jn) break;                         // (a short chunk is the last one)
                if (jn == 32 || g0 + G < jn) load_t(g0 + G < 32 ? 32 * ch + g0 + G : 32 * (ch + kUnWarps), b);
#pragma unroll
                for (int q = 0; q < G; ++q)
                    if (g0 + q < jn) {
                        const S v = conj_op ? conj(a[q]) : a[q];
#pragma unroll
                        for (int c = 0; c < RT; ++c) acc[c] += v * sq[warp][g0 + q][c];
                    }
#pragma unroll
                for (int q = 0; q < G; ++q) a[q] = b[q];
            }
            __syncwarp();
        }
        if constexpr (W == 1) {
#pragma unroll
            for (int c = 0; c < RT; ++c) {
                tot[c] = st == 0 ? acc[c] : tot[c] + acc[c];
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
            S v = nst > 0 ? ps[0][c][row] : zero<S>();
            for (int q = 1; q < nst; ++q) v = v + ps[q][c][row];
            const int64_t src = row_at(orow) + c, dst = DOWN ? src : (u.dst + orow) * nrhs + c;
            X[dst] = X[src] + v;
        }
    }
}

}  // namespace skel
