// Translations on the CUDA cores with every kernel value used twice: the
// kernels are symmetric (complex-symmetric for Helmholtz) and so is the set of
// pairs the translations evaluate, so G(t, s) serves u_t += G q_s and
// u_s += G q_t. For FP64, where the evaluation is the cost: GB300 issues 1.66 FP64
// lanes per SM and clock (measured), and a value of 3D Laplace takes 11 FP64
// operations, so an interaction with one right-hand side takes 6.5 here and 12
// in near_kernel.
//
// A warp owns an item: one target chunk (up to 32 entries of a box, one per
// lane) against up to sym_chunks() source chunks of one box (each unordered
// pair of boxes appears once). Per source chunk the lanes start at their own
// source and step through the chunk in a ring, so that in every step each
// lane evaluates another source; the sources' sums travel with them from lane
// to lane (one shuffle per step) and end at their own lane. Both sides' sums
// go to slots of 32 rows, which sym_reduce_kernel adds per chunk in a fixed
// order: the result does not depend on scheduling, and the items depend on
// the box pair only. The items run in batches that share one buffer of slots
// (kSymBatchSlots), so that its size is bounded.
// FP64, one right-hand side, near_kernel -> here (whole apply): 3D N = 2^17
// 42.4 -> 24.8 ms, N = 1,000 924 -> 53 us; 2D N = 16,384 3463 -> 530 us.
#pragma once

#include "skel_kernels.cuh"

namespace skel {

constexpr int kSymWarps = 4;

template <bool CPLX>
struct SymArgs {
    using S = typename Scal<double, CPLX>::T;
    const SymItem* items;
    int64_t n_items;
    const int64_t* chunk_start;
    const int32_t* chunk_cnt;
    const uint8_t* entry_slot;
    const double4* X;
    const S* Q;
    S* part;                               // slots x 32 rows x RT
    int nrhs, r0;
    double kappa;
    const double* logtab;                  // 2D Laplace: see log_f64
};

// ---- natural logarithm of a positive normal double ---------------------------------
// Table-driven (P.T.P. Tang, "Table-driven implementation of the logarithm
// function in IEEE arithmetic", ACM TOMS 16, 1990): x = 2^e z with
// z in [sqrt(1/2), sqrt(2)), c the table's point near z (the double 1/c is stored
// and log c is that of its exact reciprocal), f = z / c - 1 from one FMA,
// |f| < 2^-8, and
// log x = e ln 2 + log c + log1p(f) with a degree-6 series; ln 2 and log c are
// sums of a multiple of 2^-40 and a rest, so that e ln 2 + log c loses nothing.
// 13 FP64 operations (the CUDA library's log takes the time of about 27).
// Zero, subnormal and non-finite arguments go to log().
constexpr int kLogBits = 9;                // table intervals per octave (2^9)
constexpr int kLogTab = 1 << kLogBits;
constexpr int64_t kLogOff = 0x3FE6A09E667F3BCDll;   // the bits of sqrt(1/2)
__device__ __forceinline__ double log_f64(double x, const double* tab) {
    const int64_t ix = __double_as_longlong(x);
    if (ix < 0x0010000000000000ll || ix >= 0x7FF0000000000000ll) return log(x);
    const int64_t tmp = ix - kLogOff;
    const int i = (int)(tmp >> (52 - kLogBits)) & (kLogTab - 1);
    const int e = (int)(tmp >> 52);
    const double z = __longlong_as_double(ix - ((int64_t)e << 52));
    const double f = fma(z, tab[i], -1.0);
    // e as a double: an exponent that aligns the integer with the last bit
    const double ed = __longlong_as_double(0x4338000000000000ll + (int64_t)e) - 6755399441055744.0;
    constexpr double kLn2Hi = 0x1.62e42fefa2p-1;         // ln 2 to a multiple of 2^-40: e * hi is exact
    constexpr double kLn2Lo = 0x1.9ef35793c7673p-41;
    double p = fma(f, -1.0 / 6.0, 1.0 / 5.0);
    p = fma(f, p, -1.0 / 4.0);
    p = fma(f, p, 1.0 / 3.0);
    p = fma(f, p, -1.0 / 2.0);
    const double f2 = f * f;
    const double hi = fma(ed, kLn2Hi, tab[kLogTab + i]);
    const double lo = fma(ed, kLn2Lo, tab[2 * kLogTab + i]);
    return hi + (f + fma(f2, p, lo));
}

template <int KIND, int RT>
__global__ void __launch_bounds__(kSymWarps * 32) sym_kernel(const SymArgs<cplx_kind(KIND)> a) {
    using S = typename Scal<double, cplx_kind(KIND)>::T;
    using G = typename Green<double, KIND>::G;
    constexpr bool FLAT = KIND == 0 || KIND == 3;            // 2D
    __shared__ double sx[kSymWarps][3][32];
    __shared__ S sq[kSymWarps][32][RT];
    __shared__ int ss[kSymWarps][32];
    __shared__ double tab[KIND == 0 ? 3 * kLogTab : 1];
    if constexpr (KIND == 0) {
        for (int i = threadIdx.x; i < 3 * kLogTab; i += kSymWarps * 32) tab[i] = a.logtab[i];
        __syncthreads();
    }
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t id = (int64_t)blockIdx.x * kSymWarps + warp;
    if (id >= a.n_items) return;
    const SymItem it = a.items[id];
    const int64_t tst = a.chunk_start[it.tchunk];
    const int nt = a.chunk_cnt[it.tchunk];
    const bool adj = (it.flags & TASK_ADJ) != 0, self = (it.flags & kSymSelf) != 0;
    double4 tx = {0, 0, 0, 0};
    S qt[RT], at[RT];
    unsigned mrow = 0;
#pragma unroll
    for (int r = 0; r < RT; ++r) qt[r] = at[r] = zero<S>();
    if (lane < nt) {
        tx = a.X[tst + lane];
#pragma unroll
        for (int r = 0; r < RT; ++r)
            if (a.r0 + r < a.nrhs) qt[r] = a.Q[(tst + lane) * a.nrhs + a.r0 + r];
        mrow = (unsigned)(it.mask >> (8 * a.entry_slot[tst + lane])) & 0xffu;
    }
    constexpr double scale = green_scale<KIND>();
    for (int k = 0; k < it.nsrc; ++k) {
        const int64_t sst = a.chunk_start[it.schunk + k];
        const int m = a.chunk_cnt[it.schunk + k];
        __syncwarp();
        {
            double4 v = {0, 0, 0, 0};
            int slot = 0;
            if (lane < m) {
                v = a.X[sst + lane];
                slot = a.entry_slot[sst + lane];
            }
            sx[warp][0][lane] = v.x;
            sx[warp][1][lane] = v.y;
            if (!FLAT) sx[warp][2][lane] = v.z;
            ss[warp][lane] = slot;
#pragma unroll
            for (int r = 0; r < RT; ++r)
                sq[warp][lane][r] = lane < m && a.r0 + r < a.nrhs ? a.Q[(sst + lane) * a.nrhs + a.r0 + r] : zero<S>();
        }
        __syncwarp();
        // the target chunk against itself: every lane needs all sources, and
        // the sources' sums would count each pair again
        const bool diag = self && it.schunk + k == it.tchunk;
        const int M = max(nt, m);
        const int from = lane + 1 >= M ? 0 : lane + 1;
        S as[RT];
#pragma unroll
        for (int r = 0; r < RT; ++r) as[r] = zero<S>();
        int j = lane;                                        // this lane's source
#pragma unroll 4
        for (int step = 0; step < M; ++step) {
            const int js = j & 31;
            const bool on = lane < nt && j < m && !((mrow >> ss[warp][js]) & 1u);
            const double dx = tx.x - sx[warp][0][js], dy = tx.y - sx[warp][1][js];
            double r2 = dy * dy;
            if constexpr (!FLAT) {
                const double dz = tx.z - sx[warp][2][js];
                r2 = fma(dy, dy, dz * dz);
            }
            r2 = fma(dx, dx, r2);
            G g;
            if constexpr (KIND == 0) g = log_f64(r2, tab);
            else g = Green<double, KIND>::eval(r2, a.kappa);
            const bool apart = !adj || r2 > 0.0;             // coincident points contribute nothing
            if (on && apart) {
#pragma unroll
                for (int r = 0; r < RT; ++r) {
                    madd(at[r], g, sq[warp][js][r]);
                    madd(as[r], g, qt[r]);
                }
            }
#pragma unroll
            for (int r = 0; r < RT; ++r) as[r] = shfl_from(as[r], from);
            j = j + 1 >= M ? 0 : j + 1;
        }
        if (!diag) {
#pragma unroll
            for (int r = 0; r < RT; ++r) a.part[(((int64_t)it.slot + 1 + k) * 32 + lane) * RT + r] = scale * as[r];
        }
    }
#pragma unroll
    for (int r = 0; r < RT; ++r) a.part[((int64_t)it.slot * 32 + lane) * RT + r] = scale * at[r];
}

// The sums of a batch's slots, in order, to U. A warp per run (a chunk's slots of
// this batch), lane = entry; eight slots' loads in flight. The first run of a
// chunk overwrites its rows of U, the others go on from them, so the sum does
// not depend on how the items are cut into batches. Bound: HBM (the slots).
template <class S, int RT>
__global__ void __launch_bounds__(256) sym_reduce_kernel(const SymRun* __restrict__ runs, int64_t n_runs,
                                                         const int32_t* __restrict__ idx,
                                                         const int64_t* __restrict__ chunk_start,
                                                         const int32_t* __restrict__ chunk_cnt,
                                                         const S* __restrict__ part, S* __restrict__ U, int nrhs, int r0) {
    const int64_t id = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (id >= n_runs) return;
    const SymRun run = runs[id];
    const bool first = run.chunk >= 0;
    const int c = first ? run.chunk : ~run.chunk;
    const bool valid = lane < chunk_cnt[c];
    S* u = U + (chunk_start[c] + lane) * nrhs + r0;
    S sum[RT];
#pragma unroll
    for (int r = 0; r < RT; ++r) sum[r] = !first && valid && r0 + r < nrhs ? u[r] : zero<S>();
    const int64_t p1 = run.at + run.n;
    for (int64_t p = run.at; p < p1; p += 8) {
        S v[8][RT];
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const bool in = p + q < p1;
            const int64_t row = in ? ((int64_t)idx[p + q] * 32 + lane) * RT : 0;
#pragma unroll
            for (int r = 0; r < RT; ++r) v[q][r] = in ? part[row + r] : zero<S>();
        }
#pragma unroll
        for (int q = 0; q < 8; ++q)
            if (p + q < p1)
#pragma unroll
                for (int r = 0; r < RT; ++r) sum[r] += v[q][r];
    }
    if (valid) {
#pragma unroll
        for (int r = 0; r < RT; ++r)
            if (r0 + r < nrhs) u[r] = sum[r];
    }
}

}  // namespace skel
