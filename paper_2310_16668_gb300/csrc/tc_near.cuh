// On-the-fly tensor-core translations (FP32_TC, real kernels): the kernel
// values are evaluated by the CTA that multiplies them.
//
// A CTA has two groups of four compute warps (thread = row), two producer warps
// that stream pairs of tiles (chunks and descriptors) by bulk copies up to six
// pairs ahead, and two MMA warps. It owns a unit, in one of three forms:
//   * two items with consecutive rows of one box: a group each, one stream of
//     tiles for both;
//   * two unrelated items: a group each, half of the stages each;
//   * one item: each group takes 16 of a tile's 32 sources and of the 32 columns.
// In the first two a thread evaluates 32 values of a tile between hand-overs of
// a half of A, and writes one half while the tensor core works on the other:
// what a hand-over costs (mbarrier waits, fences, tensor-memory waits: about as
// long as 50 values' evaluation) is shared by many values, and an SM whose two
// CTAs are resident evaluates 1024 rows' values at a time. In the third an
// item's list ends in half the time, which counts where items are few or lists
// are short; A is then double buffered by tile.
// Bound by the evaluation's instructions (MUFU and FP32 pipes) and by what is
// left of the hand-overs. FP32, 32 right-hand sides, before (one item per CTA,
// two threads per row, three accumulating MMAs per K-step) and after: 3D,
// leaves of 128, N = 65,536 922 -> 777 us, 262,144 3988 -> 3290 us, 20,011
// 240 -> 195, 12,000 166 -> 131, 3,000 69 -> 38; 2D, leaves of 64, N = 65,536
// 252 -> 212, 3,000 66 -> 43. Plans of up to 500 points with few right-hand sides
// take up to 2 us more (N = 300, 4 right-hand sides, apply 28.7 -> 30.7).
//
// The sum, the same for all forms and for the kernels of the per-tile store (so
// all give the same bits): an item's tile list is cut into segments of 128 tiles
// (16 or 32 in small 3D plans, tc_segment) and a segment into pairs of tiles. The
// hi*hi products of a pair accumulate in
// tensor memory (D: 8 K-steps) and are then added to an FP32 register sum;
// the hi*lo and lo*hi products of the whole segment accumulate in a second
// accumulator (L), which is 2^-11 of the first in size, so that its rounding
// does not show, and is added at the segment's end. Segments are scaled and
// added in order. Of the products of a tile only four MMAs thus round at the
// size of the result (twelve did when all went into one accumulator), and a
// pair needs one read of D. B holds hi and lo as 64 columns, so hi*hi and
// hi*lo are one MMA into the adjacent columns of D and L: two MMAs per K-step
// (an issuing thread needs 48 cycles for an MMA of 32 or of 64 columns).
//
// Masks: a tile's keep word of the row's slot. A row that keeps none of 8
// sources sits at kFar (the kernel value is 0 there; 2D: multiplied by 0); where some row keeps a
// part of the 8, values are selected one by one. Chunks shorter than 32
// sources carry kFar coordinates past their end. A warp whose rows keep
// nothing of a tile writes zeros, once; a warp without valid rows takes no
// part.
#pragma once

#include <type_traits>

#include "tc_kernels.cuh"

namespace skel {

constexpr int kNearCompute = 256;              // compute threads: two groups of 128 rows
constexpr int kNearThreads = kNearCompute + 128;  // + two producer and two MMA warps
// Registers: 384 threads x 2 CTAs launch with 80 each; the compute warpgroups
// take what the last one gives up (256 x 104 + 128 x 32 = 384 x 80)
constexpr int kNearRegsCompute = 104, kNearRegsOther = 32;
static_assert(kNearCompute * kNearRegsCompute + 128 * kNearRegsOther <= kNearThreads * 80, "register split");
// a group's tensor memory (128 columns): D, L, then A in two halves of 16
// sources (hi 16 columns, lo 16 columns)
constexpr uint32_t kColNearA = 64;
// both groups on one item: D0, L, D1 (0, 32, 64), two A
constexpr uint32_t kColSplitD1 = 64, kColSplitA = 128;
constexpr int kNearPairs = 6;                  // stages of two tiles
struct alignas(128) TcPairStage {
    float chunk[2][kChunkFloats];              // B hi and lo, coordinates (hi, lo) of two tiles
    SrcTile tile[2];
};
struct TcNearShared {
    TcPairStage st[kNearPairs];
    uint64_t full[kNearPairs], empty[kNearPairs];  // per stage: copies landed; MMAs of its readers done
    uint64_t afull[2][2], done[2][2];          // per group and half of A: written; its MMAs done
    uint32_t tmem;
};
constexpr int kNearSmemRequest = 113 * 1024;   // two CTAs (2 x 256 TMEM columns) per SM
static_assert(sizeof(TcNearShared) <= kNearSmemRequest, "shared memory plan");

// Alignment of every access wider than 4 bytes (an unaligned one is a fault):
//   bulk copies, 16 bytes at both ends and in size: chunks start kChunkFloats
//     apart in a.B and in a stage, descriptors 64 bytes apart in a.tiles and in
//     tile[]; stages are 128-byte multiples of the shared memory's base;
//   mbarriers, 8 bytes: uint64_t members behind whole stages;
//   float4 reads of a chunk's coordinates: 2048 floats into the chunk, axes 32
//     floats apart, lo parts 96, sources in steps of 8, 4 per read (16 of a
//     tile's 32 sources per group: a multiple of 16 floats);
//   float4 of a.X, a.Xlo: arrays of float4;
//   float4 of U: only if nrhs is a multiple of 4, from columns that are
//     multiples of 16 (r0 of 32);
//   float4 of parts: rows of 32 floats, columns as for U;
//   float4 of stored values (fill): an item starts at abase, a multiple of 4
//     floats, and tiles are whole float4;
//   tensor-memory columns are multiples of 8, and whole warps execute every
//     tcgen05.st / ld (the waits before them end per thread: __syncwarp).
// Nothing here depends on data a bounded wait could leave stale: after one gives
// up, a descriptor may be wrong, but it only chooses among masks and flags.
static_assert(sizeof(TcPairStage) % 128 == 0 && offsetof(TcPairStage, tile) % 16 == 0, "stage layout");
static_assert(offsetof(TcNearShared, full) % 8 == 0 && offsetof(TcNearShared, tmem) % 4 == 0, "barriers");
static_assert(kChunkFloats % 4 == 0 && (2048 + 96) % 4 == 0 && sizeof(SrcTile) == 64, "chunk layout");
static_assert(sizeof(float) * kTcN % 16 == 0, "rows of partial sums");

// log of 8 squared distances. Normal arguments: x = 2^e m with m in
// [sqrt(1/2), sqrt(2)), f = m - 1 and log x = e ln 2 + (f - f^2/2 + f^3 P(f)),
// the argument reduction of S. Moshier's logf (Cephes), here by the exponent bits
// relative to those of sqrt(1/2); P of degree 7 fitted to
// (log(1 + f) - f + f^2/2) / f^3 on that interval (against 64 bits: within 8e-9 of
// the logarithm), ln 2 as a sum of two floats the first of which has 9
// significant bits (as there): within 0.9 ulp, half
// the instructions of logf because two values share each. on: 1, or 0 for a row
// that keeps none of these sources. ADJ: subnormal x (whose exponent field says
// nothing) go to logf; 0 for x = 0 if the leaves touch.
template <bool ADJ>
__device__ __forceinline__ void tc_log8(const float* r2, float on, bool touch, float* g) {
    auto f2 = [](float v) { return make_float2(v, v); };
    const float2 on2 = f2(on);
#pragma unroll
    for (int j = 0; j < 8; j += 2) {
        int ix = __float_as_int(r2[j]), iy = __float_as_int(r2[j + 1]);
        // (nvcc 13.0 gives a wrong first result when the halves of a paired
        // FP32 result are used as integers without a copy in between)
        asm volatile("" : "+r"(ix), "+r"(iy));
        const int ex = (ix - 0x3f3504f3) >> 23, ey = (iy - 0x3f3504f3) >> 23;
        const float2 f = __fadd2_rn(make_float2(__int_as_float(ix - (ex << 23)), __int_as_float(iy - (ey << 23))), f2(-1.f));
        // e as a float: added to the bits of 1.5 * 2^23
        const float2 e = __fadd2_rn(make_float2(__int_as_float(0x4B400000 + ex), __int_as_float(0x4B400000 + ey)),
                                    f2(-12582912.f));
        const float2 z = __fmul2_rn(f, f);
        float2 q = __ffma2_rn(f, f2(-0.0785954595f), f2(0.128816217f));
        q = __ffma2_rn(f, q, f2(-0.131287679f));
        q = __ffma2_rn(f, q, f2(0.141811967f));
        q = __ffma2_rn(f, q, f2(-0.166245535f));
        q = __ffma2_rn(f, q, f2(0.200022861f));
        q = __ffma2_rn(f, q, f2(-0.250008106f));
        q = __ffma2_rn(f, q, f2(0.333333164f));
        q = __fmul2_rn(__fmul2_rn(f, z), q);
        q = __ffma2_rn(z, f2(-0.5f), q);
        q = __ffma2_rn(e, f2((float)(0.693147180559945309417 - 0.693359375)), q);
        q = __ffma2_rn(e, f2(0.693359375f), __fadd2_rn(f, q));
        q = __fmul2_rn(q, on2);
        g[j] = q.x;
        g[j + 1] = q.y;
    }
    if (ADJ) {
        float lo = r2[0];
#pragma unroll
        for (int j = 1; j < 8; ++j) lo = fminf(lo, r2[j]);
        // (the warp stays together: tensor-memory stores follow)
        if (__any_sync(0xffffffffu, lo < 1.17549435e-38f)) {
#pragma unroll
            for (int j = 0; j < 8; ++j)
                if (r2[j] < 1.17549435e-38f) g[j] = !touch || r2[j] > 0.f ? on * logf(r2[j]) : 0.f;
            __syncwarp();
        }
    }
}

// 8 sources (coordinates at x: 32 floats per axis; lo parts 96 floats on)
// against this thread's target, two sources per paired FP32 instruction: the
// kernel values in g, not masked. nt, nl: the negated target. touch: of two
// touching leaves.
template <int KIND, bool ADJ>
__device__ __forceinline__ void tc_eval8(const float* x, float4 nt, float4 nl, bool touch, float* g) {
    constexpr int AX = 32, LO = 96;
    const float2 ntx = make_float2(nt.x, nt.x), nty = make_float2(nt.y, nt.y), ntz = make_float2(nt.z, nt.z);
    float d2[KIND == 0 ? 8 : 1];
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        const float4 X = *reinterpret_cast<const float4*>(x + 4 * q);
        const float4 Y = *reinterpret_cast<const float4*>(x + AX + 4 * q);
        float4 Z, LX, LY, LZ;
        if (KIND != 0) Z = *reinterpret_cast<const float4*>(x + 2 * AX + 4 * q);
        if (ADJ) {
            LX = *reinterpret_cast<const float4*>(x + LO + 4 * q);
            LY = *reinterpret_cast<const float4*>(x + LO + AX + 4 * q);
            if (KIND != 0) LZ = *reinterpret_cast<const float4*>(x + LO + 2 * AX + 4 * q);
        }
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            float2 dx = __fadd2_rn(h ? make_float2(X.z, X.w) : make_float2(X.x, X.y), ntx);
            float2 dy = __fadd2_rn(h ? make_float2(Y.z, Y.w) : make_float2(Y.x, Y.y), nty);
            if (ADJ) {
                dx = __fadd2_rn(dx, __fadd2_rn(h ? make_float2(LX.z, LX.w) : make_float2(LX.x, LX.y),
                                               make_float2(nl.x, nl.x)));
                dy = __fadd2_rn(dy, __fadd2_rn(h ? make_float2(LY.z, LY.w) : make_float2(LY.x, LY.y),
                                               make_float2(nl.y, nl.y)));
            }
            float2 r2 = __fmul2_rn(dx, dx);
            r2 = __ffma2_rn(dy, dy, r2);
            if (KIND != 0) {
                float2 dz = __fadd2_rn(h ? make_float2(Z.z, Z.w) : make_float2(Z.x, Z.y), ntz);
                if (ADJ)
                    dz = __fadd2_rn(dz, __fadd2_rn(h ? make_float2(LZ.z, LZ.w) : make_float2(LZ.x, LZ.y),
                                                   make_float2(nl.z, nl.z)));
                r2 = __ffma2_rn(dz, dz, r2);
            }
            if constexpr (KIND == 0) {
                d2[4 * q + 2 * h] = r2.x;
                d2[4 * q + 2 * h + 1] = r2.y;
            } else {
                g[4 * q + 2 * h] = tc_rsqrt<ADJ>(r2.x);
                g[4 * q + 2 * h + 1] = tc_rsqrt<ADJ>(r2.y);
            }
        }
    }
    if constexpr (KIND == 0) tc_log8<ADJ>(d2, nt.x < kFar ? 1.f : 0.f, touch, g);
}

// Veltkamp's split of 8 values into TF32 hi and lo: hi = t - (t - g) with
// t = (2^13 + 1) g keeps 11 significant bits of g (a TF32 value, rounded to
// nearest); lo = g - hi is exact. hi goes to the 8 tensor-memory columns from
// taddr, lo to those 16 columns on.
__device__ __forceinline__ void tc_split_store(const float* g, uint32_t taddr) {
    const float2 m1 = make_float2(-1.f, -1.f), split = make_float2(8193.f, 8193.f);
    uint32_t hi[8], lo[8];
#pragma unroll
    for (int j = 0; j < 8; j += 2) {
        const float2 v = make_float2(g[j], g[j + 1]);
        const float2 t = __fmul2_rn(v, split);
        const float2 h = __ffma2_rn(__ffma2_rn(v, m1, t), m1, t);
        const float2 l = __ffma2_rn(h, m1, v);
        hi[j] = __float_as_uint(h.x);
        hi[j + 1] = __float_as_uint(h.y);
        lo[j] = __float_as_uint(l.x);
        lo[j + 1] = __float_as_uint(l.y);
    }
    tmem_st8(taddr, hi);
    tmem_st8(taddr + 16u, lo);
}

// a += the 16 (32) tensor-memory columns from taddr of this thread's lane
__device__ __forceinline__ void tmem_add16(uint32_t taddr, float2* a) {
    uint32_t v[16];
    tmem_ld16(taddr, v);
#pragma unroll
    for (int c = 0; c < 8; ++c)
        a[c] = __fadd2_rn(a[c], make_float2(__uint_as_float(v[2 * c]), __uint_as_float(v[2 * c + 1])));
}
__device__ __forceinline__ void tmem_add32(uint32_t taddr, float2* a) {
    uint32_t v[32];
    tmem_ld16(taddr, v);
    tmem_ld16(taddr + 16u, v + 16);
#pragma unroll
    for (int c = 0; c < 16; ++c)
        a[c] = __fadd2_rn(a[c], make_float2(__uint_as_float(v[2 * c]), __uint_as_float(v[2 * c + 1])));
}

template <int N>
__device__ __forceinline__ void tmem_zero(uint32_t taddr) {
    uint32_t z[8];
#pragma unroll
    for (int c = 0; c < 8; ++c) z[c] = 0u;
#pragma unroll
    for (int c = 0; c < N; c += 8) tmem_st8(taddr + c, z);
}

// REC: the fill pass of a stored-operator mode also writes the kernel values
// it evaluates to a.A: kRecTiles every tile's values as the MMA consumes them
// (masked), kRecSym the blocks this tile records for the symmetric store
// (every source of the chunk, unmasked). Fill passes run one item per unit.
constexpr int kRecNone = 0, kRecTiles = 1, kRecSym = 2;

// one thread's targets and masks for a tile
struct TcNearRow {
    float4 x, lo;                              // coordinates (hi, lo)
    int slot;                                  // its slot of the item
    bool valid;
};
struct TcNearTile {
    float4 nt, nl;                             // negated target: in the frame of the chunk; lo parts
    uint32_t kw;                               // kept sources
    bool none, some;                           // warp: no row keeps any source; some row keeps a part
};
template <int REC>
__device__ __forceinline__ TcNearTile tc_near_tile(const TcNearRow& r, const SrcTile& st, uint32_t all, bool adj,
                                                   int first) {
    TcNearTile t;
    t.kw = r.valid ? st.keep[r.slot] >> first & all : 0u;  // of the thread's sources, from source `first`
    t.none = REC == kRecNone && __all_sync(0xffffffffu, t.kw == 0u);
    t.some = REC != kRecSym && __any_sync(0xffffffffu, t.kw != 0u && t.kw != all);
    tc_frame(r.x, r.lo, st.cen, adj, t.nt, t.nl);
    if (REC != kRecSym && t.kw == 0u) t.nt.x = kFar;
    return t;
}
// masks of 8 sources q: this row's target moved to kFar if it keeps none of
// them; true if some row of the warp keeps a part of them
__device__ __forceinline__ bool tc_near_cut(const TcNearTile& t, uint32_t all, int q, float4& at) {
    at = t.nt;
    if (!t.some) return false;
    const uint32_t kb = t.kw >> (8 * q) & 0xFFu;
    if (kb == 0u) at.x = kFar;
    return __any_sync(0xffffffffu, kb != 0u && kb != (all >> (8 * q) & 0xFFu));
}
__device__ __forceinline__ void tc_near_select(const TcNearTile& t, int q, float* g) {
    const uint32_t kb = t.kw >> (8 * q);
#pragma unroll
    for (int j = 0; j < 8; ++j) g[j] = (kb >> j) & 1u ? g[j] : 0.f;
}

// The compute warps of one group: thread = row of an item.
// Its tiles come in np stages from stage `ring`.
// SPLIT = false: the group has its own item, all 32 sources of a tile and its
// own columns of tensor memory; A's halves b = 0, 1 are handed over in turn.
// SPLIT = true: both groups have the same item, group g the half g of every
// tile's sources and the columns 16 g .. 16 g + 15 of the sums; A is double
// buffered by tile (buffer t % 2), and pairs alternate between two D (columns
// 0 and 64), so that nobody waits for the MMAs of the pair just handed over.
// parts: where the segments of a cut item go (null: to U).
template <int KIND, int REC, bool SPLIT>
__device__ __forceinline__ bool tc_near_rows(const TcArgs& a, TcNearShared& S, int ring, int np, int g, int item,
                                             int t_lo, int t_hi, float* parts, int rot, uint32_t tbase) {
    constexpr int NC = SPLIT ? 16 : 32;                    // accumulator columns of a thread
    const int warp = (threadIdx.x >> 5) & 3, lane = threadIdx.x & 31;
    const TcItem* itp = a.items + item;
    const int nrows = itp->nrows, list_lo = itp->list_lo, lseg = itp->lseg;
    // warp w always runs on scheduler w % 4: the 32-row blocks are dealt to the
    // warps from a position that moves with the CTA
    const int blk = (warp + rot) & 3, row = 32 * blk + lane;
    if (32 * blk >= nrows) return true;
    const uint32_t base = tbase + ((uint32_t)(warp * 32) << 16) + (SPLIT ? 0u : 128u * g);
    const uint32_t dcol = base + (SPLIT ? 16u * g : 0u), lcol = dcol + 32u;
    const uint32_t acol = base + (SPLIT ? kColSplitA + 32u * g : kColNearA);
    TcNearRow rw;
    rw.valid = row < nrows;
    const int64_t urow = itp->row_off + row;
    rw.slot = 0;
    for (int c = 1; c < itp->nslot; ++c)
        if (row >= itp->slot_start[c]) rw.slot = c;
    rw.x = rw.lo = make_float4(0.f, 0.f, 0.f, 0.f);
    if (rw.valid) {
        rw.x = a.X[urow];
        rw.lo = a.Xlo[urow];
    }
    // fill passes: this row's row chunk and its row in it; the floats of the
    // tiles before the current one
    int rk = 0, rl = row, rm = 1;
    int64_t rref0 = 0, tfill = 0;
    if constexpr (REC == kRecSym) {
        const ItemSym* is = a.isym + item;
        rm = is->m;
        rref0 = is->ref0;
        for (int k = 1; k < rm; ++k)
            if (row >= is->ro[k]) rk = k;
        rl = row - is->ro[rk];
    }
    bool ok = true;
    uint32_t cnt = 0u;                                     // tiles handed over: the phases of afull and done
    // the MMAs of the previous tile's half b (SPLIT: of tile cnt - back) are done
    auto wait_done = [&](int b, uint32_t back) {
        if constexpr (SPLIT) {
            if (cnt >= back) {
                const uint32_t t = cnt - back;
                ok &= mbar_wait_warp(sm_addr(&S.done[t & 1u][0]), (t >> 1) & 1u, a.wait_ns);
            }
        } else {
            if (cnt > 0u) ok &= mbar_wait_warp(sm_addr(&S.done[g][b]), (cnt - 1u) & 1u, a.wait_ns);
        }
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    };
    auto hand_over = [&](int b) {
        asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncwarp();
        if (lane == 0) mbar_arrive(sm_addr(SPLIT ? &S.afull[cnt & 1u][g] : &S.afull[g][b]));
    };
    auto sum = [&](uint32_t taddr, float2* acc) {
        if constexpr (SPLIT) tmem_add16(taddr, acc);
        else tmem_add32(taddr, acc);
    };
    float2 acc[NC / 2];
    uint32_t azero = 0u;                                   // A (SPLIT: bit per buffer) holds zeros in this warp's rows
    int s = 0;
    uint32_t ph = 0u;
    int s0 = t_lo;
    do {                                                   // segments (an item without tiles writes zeros)
        const int send = min(s0 + (1 << lseg), t_hi);
#pragma unroll
        for (int c = 0; c < NC / 2; ++c) acc[c] = make_float2(0.f, 0.f);
        __syncwarp();                                      // (rows that are not valid skipped the end of a segment)
        tmem_zero<NC>(dcol);
        tmem_zero<NC>(lcol);
        if (SPLIT) tmem_zero<NC>(dcol + kColSplitD1);
        for (int t = s0; t < send; ++t) {
            const int ti = t & 1;
            const TcPairStage& st = S.st[ring + s];
            if (ti == 0) ok &= mbar_wait_warp(sm_addr(&S.full[ring + s]), ph, a.wait_ns);
            const SrcTile& tl = st.tile[ti];
            const float* xs = st.chunk[ti] + 2048;
            // touching leaves take the form with lo parts and guards, and so do
            // the other boxes of a 2D plan so small that their r^2 may be
            // subnormal (guards in the other form cost every 2D plan 13% of
            // this kernel: N = 65,536 218 -> 246 us)
            const bool touch = (tl.flags & TASK_ADJ) != 0;
            const bool adj = touch || (KIND == 0 && a.subnormal);
            uint32_t all = tl.cnt >= 32 ? 0xFFFFFFFFu : (1u << (tl.cnt & 31)) - 1u;
            if (SPLIT) all = all >> (16 * g) & 0xFFFFu;
            const TcNearTile ta = tc_near_tile<REC>(rw, tl, all, adj, SPLIT ? 16 * g : 0);
            const uint32_t at_col = acol + (SPLIT ? 64u * (uint32_t)ti : 0u);
            const uint32_t abit = SPLIT ? 1u << ti : 1u;
            // before the first MMAs of a pair: the pair that its D held (SPLIT:
            // the pair two before it, whose MMAs wait_done(0, 2) has waited for)
            auto drain = [&]() {
                if constexpr (SPLIT) {
                    if (ti == 0 && t >= s0 + 4) {
                        const uint32_t dc = dcol + (t & 2 ? kColSplitD1 : 0u);
                        sum(dc, acc);
                        tmem_zero<NC>(dc);
                    }
                } else if (ti == 0 && t > s0) {
                    wait_done(1, 1u);
                    sum(dcol, acc);
                    tmem_zero<NC>(dcol);
                }
            };
            if (ta.none) {
#pragma unroll
                for (int b = 0; b < (SPLIT ? 1 : 2); ++b) {
                    wait_done(b, 2u);
                    if (!(azero & abit)) tmem_zero<32>(at_col + 32u * b);
                    if (b == 0) drain();
                    hand_over(b);
                }
                azero |= abit;
            } else {
                azero &= ~abit;
                // CUT: some row keeps a part of the sources
                auto tile = [&](auto ADJ, auto CUT) {
#pragma unroll
                    for (int b = 0; b < (SPLIT ? 1 : 2); ++b) {
#pragma unroll
                        for (int e = 0; e < 2; ++e) {
                            const int q = 2 * b + e;                     // 8 sources of the thread's
                            const float* xq = xs + 8 * q + (SPLIT ? 16 * g : 0);
                            [[maybe_unused]] const int tq = q + (SPLIT ? 2 * g : 0);   // of the tile's
                            float gv[8];
                            float4 at = ta.nt;
                            bool cut = false;
                            if constexpr (decltype(CUT)::value) cut = tc_near_cut(ta, all, q, at);
                            tc_eval8<KIND, decltype(ADJ)::value>(xq, at, ta.nl, touch, gv);
                            if constexpr (REC == kRecSym) {
                                // this row's block of the tile, if this tile records it
                                // (stored as this row chunk x the tile's chunk)
                                const BlockRef rf = a.refs[rref0 + (int64_t)t * rm + rk];
                                if (rw.valid && (rf.flags & kRefRecord)) {
#pragma unroll
                                    for (int j = 0; j < 8; ++j)
                                        if (8 * tq + j < tl.cnt)
                                            a.A[rf.off + (int64_t)(8 * tq + j) * rf.pitch + rl] = gv[j];
                                }
                            }
                            if (cut) tc_near_select(ta, q, gv);
                            if constexpr (REC == kRecTiles) {
                                const uint32_t qm = a.qmask[list_lo + t];
                                float4* dst = reinterpret_cast<float4*>(a.A + a.abase[item] + tfill);
#pragma unroll
                                for (int h = 0; h < 2; ++h)
                                    if (rw.valid && ((qm >> (2 * tq + h)) & 1u))
                                        dst[tile_word(qm, 2 * tq + h, row, nrows)] =
                                            make_float4(gv[4 * h], gv[4 * h + 1], gv[4 * h + 2], gv[4 * h + 3]);
                            }
                            if (e == 0) wait_done(b, 2u);
                            tc_split_store(gv, at_col + 32u * b + 8u * e);
                        }
                        if (b == 0) drain();
                        hand_over(b);
                    }
                };
                if (ta.some) {
                    if (adj) tile(std::true_type{}, std::true_type{});
                    else tile(std::false_type{}, std::true_type{});
                } else {
                    if (adj) tile(std::true_type{}, std::false_type{});
                    else tile(std::false_type{}, std::false_type{});
                }
                if constexpr (REC == kRecTiles) tfill += (int64_t)__popc((uint32_t)a.qmask[list_lo + t]) * nrows * 4;
            }
            ++cnt;
            if ((ti == 1 || t == send - 1) && ++s == np) s = 0, ph ^= 1u;
        }
        if (send > s0) {
            // the last pair, then the segment's small products
            wait_done(0, 2u);
            wait_done(1, 1u);
            if constexpr (SPLIT) {
                const int np = (send - s0 + 1) / 2;        // a segment starts with D0
                for (int p = max(np - 2, 0); p < np; ++p) sum(dcol + (p & 1 ? kColSplitD1 : 0u), acc);
            } else {
                sum(dcol, acc);
            }
            sum(lcol, acc);
        }
        if (rw.valid) {
            float v[NC];
#pragma unroll
            for (int c = 0; c < NC / 2; ++c) v[2 * c] = acc[c].x, v[2 * c + 1] = acc[c].y;
            const int c0 = SPLIT ? 16 * g : 0;
            if (parts == nullptr) {
                tc_add_rows<KIND, NC>(a, urow, c0, s0 > 0, v);
            } else {
                // a part of the item: its segments go to their own rows
                float4* d = reinterpret_cast<float4*>(parts + ((int64_t)(s0 >> lseg) * kTcRows + row) * kTcN + c0);
#pragma unroll
                for (int c = 0; c < NC / 4; ++c) d[c] = make_float4(v[4 * c], v[4 * c + 1], v[4 * c + 2], v[4 * c + 3]);
            }
        }
        s0 += 1 << lseg;
    } while (s0 < t_hi);
    return ok;
}

template <int KIND, int REC = kRecNone>
__global__ void __launch_bounds__(kNearThreads, 2) tc_near_kernel(const TcArgs a) {
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    TcNearShared& S = *reinterpret_cast<TcNearShared*>(smem_raw);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const TcUnit un = a.units[blockIdx.x];
    // two items, with one stream of tiles for both or one each; or one item
    const bool two = un.b >= 0, streams = two && !un.shared;
    const int np = streams ? kNearPairs / 2 : kNearPairs;
    // the tiles of group g's item this unit covers
    auto t_lo = [&](int g) { return g ? un.lo_b : un.lo_a; };
    auto t_hi = [&](int g) {
        const TcItem& it = a.items[g ? un.b : un.a];
        return min(t_lo(g) + un.count, it.list_hi - it.list_lo);
    };

    if (tid == 0) {
        for (int s = 0; s < kNearPairs; ++s) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" :: "r"(sm_addr(&S.full[s])));
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;"
                         :: "r"(sm_addr(&S.empty[s])), "r"(two && un.shared ? 2 : 1));
        }
        for (int i = 0; i < 2; ++i)
            for (int j = 0; j < 2; ++j) {
                // the warps that hold rows (the others take no part)
                const int warps = (a.items[two && i ? un.b : un.a].nrows + 31) / 32;
                asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" :: "r"(sm_addr(&S.afull[i][j])), "r"(warps));
                asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" :: "r"(sm_addr(&S.done[i][j])));
            }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     :: "r"(sm_addr(&S.tmem)), "r"(kTmemCols));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tbase = S.tmem;
    bool err = false;

    if (warp >= kNearCompute / 32) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" :: "n"(kNearRegsOther));
        const int role = warp - kNearCompute / 32;           // 0, 1: producers; 2, 3: MMA issuers of the groups
        const int g = role & 1;
        const int item = two && g ? un.b : un.a;
        const int ring = streams ? g * np : 0;
        const int list_lo = a.items[item].list_lo + t_lo(two ? g : 0), ntile = t_hi(two ? g : 0) - t_lo(two ? g : 0);
        if (role == 0 || (role == 1 && streams)) {
            // ---------------- producer: bulk copies up to np pairs ahead ----------------
            const bool hold = item == a.withhold_item;
            const int npair = (ntile + 1) / 2;
            int s = 0;
            uint32_t ph = 1u;                                // phase of empty (not waited for in the first round)
            for (int p0 = 0; p0 < npair; p0 += 16) {
                const int my_chunk = 2 * p0 + lane < ntile ? a.tiles[list_lo + 2 * p0 + lane].chunk : 0;
                const int n = min(16, npair - p0);
                for (int i = 0; i < n; ++i) {
                    const int p = p0 + i;
                    const int c0 = __shfl_sync(0xffffffffu, my_chunk, 2 * i);
                    const int c1 = __shfl_sync(0xffffffffu, my_chunk, 2 * i + 1);
                    const bool both = 2 * p + 1 < ntile;
                    if (p >= np && !mbar_wait(sm_addr(&S.empty[ring + s]), ph, a.wait_ns)) err = true;
                    if (hold && p == 0 && !withhold_first_tile(sm_addr(&S.afull[two ? g : 0][0]), a.wait_ns)) err = true;
                    if (lane == 0) {
                        TcPairStage& st = S.st[ring + s];
                        const uint32_t bar = sm_addr(&S.full[ring + s]);
                        const uint64_t keep = l2_evict_last();
                        mbar_arrive_tx(bar, (both ? 2u : 1u) * (4u * kChunkFloats + 64u));
                        bulk_g2s_hint(sm_addr(st.chunk[0]), a.B + (int64_t)c0 * kChunkFloats, 4u * kChunkFloats, bar, keep);
                        if (both)
                            bulk_g2s_hint(sm_addr(st.chunk[1]), a.B + (int64_t)c1 * kChunkFloats, 4u * kChunkFloats, bar,
                                          keep);
                        bulk_g2s_hint(sm_addr(st.tile), a.tiles + list_lo + 2 * p, both ? 128u : 64u, bar,
                                      l2_evict_first());
                        // (after a withheld tile the compute warps may run ahead of
                        // the copies: each stage lands before it is armed again)
                        if (hold && !mbar_wait(bar, ph ^ 1u, a.wait_ns)) err = true;
                    }
                    __syncwarp();
                    if (++s == np) s = 0, ph ^= 1u;
                }
            }
            if (lane == 0) {
                // all bulk copies have landed and all commits have arrived
                // before the CTA may exit
                for (int p = max(npair - np, 0); p < npair; ++p) {
                    const uint32_t par = (uint32_t)(p / np) & 1u;
                    if (!mbar_wait(sm_addr(&S.full[ring + p % np]), par, a.wait_ns)) err = true;
                    if (!mbar_wait(sm_addr(&S.empty[ring + p % np]), par, a.wait_ns)) err = true;
                }
            }
        } else if (role == 2 || (role == 3 && two)) {
            // ---------------- MMA issuers (one thread per group; both groups' item: one) ----------------
            if (lane == 0) {
                const uint32_t idesc32 =
                    (1u << 4) | (2u << 7) | (2u << 10) | ((uint32_t)(kTcN >> 3) << 17) | ((128u >> 4) << 24);
                const uint32_t idesc64 =
                    (1u << 4) | (2u << 7) | (2u << 10) | ((uint32_t)(2 * kTcN >> 3) << 17) | ((128u >> 4) << 24);
                auto commit = [&](uint64_t* bar) {
                    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];"
                                 :: "r"(sm_addr(bar)) : "memory");
                };
                auto wait_a = [&](uint64_t* bar, uint32_t parity) {
                    if (!mbar_wait(sm_addr(bar), parity, a.wait_ns)) err = true;
                };
                const uint32_t dcol = tbase + 128u * g;
                // D, L += hi [hi | lo]; L += lo hi for the 16 sources of half b of the A operand at acol
                // (d1: the D that is not next to L, two MMAs instead of the first)
                auto half = [&](uint32_t acol, uint32_t b0, int b, bool d1) {
#pragma unroll
                    for (int k = 0; k < 2; ++k) {
                        const uint32_t desc = b0 + kDescStep * (2 * b + k), ac = acol + 32u * b + 8u * k;
                        if (d1) {
                            mma_tf32_lo(dcol + kColSplitD1, ac, desc, idesc32, true);
                            mma_tf32_lo(dcol + 32u, ac, desc + kDescLoPart, idesc32, true);
                        } else {
                            mma_tf32_lo(dcol, ac, desc, idesc64, true);
                        }
                        mma_tf32_lo(dcol + 32u, ac + 16u, desc, idesc32, true);
                    }
                };
                int s = 0;
                for (int t = 0; t < ntile; ++t) {
                    const uint32_t b0 = smem_desc_lo(sm_addr(S.st[ring + s].chunk[t & 1]));
                    const bool last = (t & 1) || t == ntile - 1;   // of its pair
                    if (two) {
#pragma unroll
                        for (int b = 0; b < 2; ++b) {
                            wait_a(&S.afull[g][b], (uint32_t)t & 1u);
                            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                            half(dcol + kColNearA, b0, b, false);
                            if (b == 1 && last) commit(&S.empty[ring + s]);
                            commit(&S.done[g][b]);
                        }
                    } else {
                        // both halves first: each group adds and clears its
                        // columns of D before it hands over the first tile of a pair
                        const uint32_t acol = dcol + kColSplitA + 64u * (uint32_t)(t & 1);
                        wait_a(&S.afull[t & 1][0], (uint32_t)(t >> 1) & 1u);
                        wait_a(&S.afull[t & 1][1], (uint32_t)(t >> 1) & 1u);
                        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                        half(acol, b0, 0, (t & 2) != 0);
                        half(acol, b0, 1, (t & 2) != 0);
                        if (last) commit(&S.empty[ring + s]);
                        commit(&S.done[t & 1][0]);
                    }
                    if (last && ++s == np) s = 0;
                }
            }
        }
    } else {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" :: "n"(kNearRegsCompute));
        const int g = warp >> 2;
        const int item = two && g ? un.b : un.a;
        const int lo = t_lo(two ? g : 0), hi = t_hi(two ? g : 0);
        float* parts = nullptr;
        if (a.parts != nullptr && a.part0[item] >= 0) parts = a.parts + a.part0[item] * (kTcRows * kTcN);
        const int rot = (int)(blockIdx.x + (two ? 2u * (uint32_t)g : 0u));
        bool ok;
        if constexpr (REC == kRecNone)
            ok = two ? tc_near_rows<KIND, REC, false>(a, S, streams ? g * np : 0, np, g, item, lo, hi, parts, rot, tbase)
                     : tc_near_rows<KIND, REC, true>(a, S, 0, np, g, item, lo, hi, parts, rot, tbase);
        else
            ok = tc_near_rows<KIND, REC, true>(a, S, 0, np, g, item, lo, hi, parts, rot, tbase);
        if (!ok) err = true;
    }
    if (err) atomicExch(a.status, 1);
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 0) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" :: "r"(tbase), "r"(kTmemCols));
    }
}

// The items whose lists were cut over several units: U = the sum of their
// segments, in order (one CTA per item; a thread owns 4 columns of a row).
// The scaling and the order of the additions are those of tc_add_rows.
template <int KIND>
__global__ void __launch_bounds__(256) tc_segments_kernel(const TcArgs a, const int32_t* __restrict__ split) {
    const int item = split[blockIdx.x];
    const TcItem it = a.items[item];
    const int nseg = (it.list_hi - it.list_lo + (1 << it.lseg) - 1) >> it.lseg;
    const float scale = (float)green_scale<KIND>();
    const float* parts = a.parts + a.part0[item] * (kTcRows * kTcN);
    for (int i = threadIdx.x; i < it.nrows * (kTcN / 4); i += 256) {
        const int row = i / (kTcN / 4), c0 = 4 * (i % (kTcN / 4));
        float4 u = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 4
        for (int s = 0; s < nseg; ++s) {
            const float4 v = *reinterpret_cast<const float4*>(parts + ((int64_t)s * kTcRows + row) * kTcN + c0);
            const float4 w = make_float4(__fmul_rn(scale, v.x), __fmul_rn(scale, v.y), __fmul_rn(scale, v.z),
                                         __fmul_rn(scale, v.w));
            u = s == 0 ? w : make_float4(__fadd_rn(u.x, w.x), __fadd_rn(u.y, w.y), __fadd_rn(u.z, w.z),
                                         __fadd_rn(u.w, w.w));
        }
        float* d = a.U + (it.row_off + row) * a.nrhs + a.r0 + c0;
        const float* uv = &u.x;
#pragma unroll
        for (int c = 0; c < 4; ++c)
            if (a.r0 + c0 + c < a.nrhs) d[c] = uv[c];
    }
}

}  // namespace skel
