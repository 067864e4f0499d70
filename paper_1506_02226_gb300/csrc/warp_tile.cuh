// warp_tile.cuh — the exact pair test of ordered rows for d <= 16, a warp at a
// time on matrix instructions, and the passes built on it: many instances at
// once (batch.cu) and one instance's all-pairs run (pairs_wt.cu).
//
// Rows hold centred units v = u - 512 in [-512, 511] as FP16 (exact), padded
// to 16 coordinates, so one mma.sync m16n8k16 gives the dot products of 16 x 8
// pairs.  Exactness: every product and every partial sum of G = v_p . v_q is
// an integer of magnitude <= 16 * 2^18 = 2^22, so the FP32 accumulator holds G
// exactly in any order of addition; the score T + 1 - |p|^2 - |q|^2 + 2 G is
// then formed in FP32 as (2 G - |q|^2) + (T + 1 - |p|^2), both integers of
// magnitude below 2^24, and so is their sum T + 1 - D: the decision score >= 1
// is exact, as in the scalar form (ap_tile.cuh).  (mma.sync and not tcgen05: a
// work item here is a few 32 x 64 pair blocks of one small instance, and a
// fragment in registers needs no staging, no barrier and no tensor memory.)
// SIMT forms of the kernels take the same sums on the CUDA cores in FP32.
//
// Work.  A tile is 64 consecutive rows of one instance, in an order that puts
// close rows next to each other; a work item is half a tile (32 rows, its
// operand fragments held in registers) against a range of column tiles, and
// belongs to one warp: a warp never waits for another.  Most column tiles need
// no score:
//   box    the tiles' boxes (least and greatest unit per axis) lie more than
//          eps apart: no neighbour pair (32 tiles tested at once, a lane each);
//   count  once all 32 rows have min_pts neighbours, counted from their own
//          tile outwards, their counts no longer matter;
//   merge  each tile's core rows are joined among themselves when its core
//          flags are set (core_tile, in shared memory), so the merge only
//          crosses tiles; it takes the next kNear tiles first, then skips every
//          pair of tiles whose core rows are known to be one set (the tags);
//          one hit joins two tiles that are one set each;
//   border only rows that are not core and have a neighbour at all look for
//          one; only tiles with core rows are looked at.
// Rows, tiles and forest are indexed over the whole batch (row = 64 tile + r),
// so an item needs one record and no per-instance pointers.
#pragma once

#include <cuda_fp16.h>

#include <climits>

#include "batch_items.h"
#include "internal.cuh"

namespace wtile {

constexpr int BT = 64, NT = 256;  // rows per tile, threads per block
constexpr int kNear = 2;          // merge: column tiles right after the row tile, taken first
constexpr unsigned FULL = 0xffffffffu;
enum { WT_COUNT = 0, WT_NEAR = 1, WT_FAR = 2, WT_BORDER = 3 };
constexpr int kNoCore = -2, kMixed = -1;  // tags: no core row, core rows of several sets (else their root)

// What a work item needs of its instance, one record per tile.
struct __align__(16) TileRec {
    int tile0, ntiles;  // the instance's tiles
    int n, d;
    int Tc, min_pts;
    float Tp1;
    int inst;
    int point0;         // the instance's first point in point-indexed arrays
    int leave;          // count: rows stop mattering at this many neighbours (min_pts, or INT_MAX: exact counts)
    int pad[2];
};

struct Hdr {  // device-side sizes of a run
    int count;        // instances
    int total_points;
    int total_tiles;
    int max_chunks;   // column chunks of the largest instance
};

struct Rows {  // by row of the batch (64 per tile), unless said otherwise
    const TileRec *tiles;  // by tile
    const uint2 *P16;      // four pieces a row: piece k holds units 2k, 2k+1, 2k+8, 2k+9
    const float *nb;       // -|v|^2 (-1e30 past an instance's last row)
    float *nbc;            // the same for core rows, -1e30 for the others
    const float *box;      // least unit of every tile on axis k at [k * cap_tiles], greatest at [(16 + k) * cap_tiles]
    long long cap_tiles;
    int *count;
    uint8_t *core;
    int *parent;
    int *border;           // smallest-index core neighbour (a point)
    const int *perm;       // point of each row
    int *tag, *need;       // by tile: common root of its core rows; some row needs the border pass
    unsigned *status;
    unsigned long long *ev;  // pair tests evaluated, three per instance: count, merge, border (nullable)
};

// 16 x 8 dot products over 16 coordinates.
__device__ __forceinline__ void mma16(float (&c)[4], const unsigned (&a)[4], uint2 b) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%10,%11,%12,%13};"
        : "=f"(c[0]), "=f"(c[1]), "=f"(c[2]), "=f"(c[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b.x), "r"(b.y), "f"(0.f), "f"(0.f), "f"(0.f), "f"(0.f));
}
// The same products on the CUDA cores, in FP32 (a batch whose plan asks for
// DBSCAN_PREC_EXACT_SIMT): the fragments' units are fetched from the lanes that
// hold them, four at a time for each of the lane's two rows and two columns.
__device__ __forceinline__ void fma16(float (&c)[4], const unsigned (&a)[4], uint2 b) {
    const int lane = threadIdx.x & 31;
    auto f2 = [](unsigned v) { return __half22float2(*reinterpret_cast<const __half2 *>(&v)); };
    c[0] = c[1] = c[2] = c[3] = 0.f;
#pragma unroll 1  // unrolled, the rows' units of a whole tile are held at once and spill (a kilobyte in the count)
    for (int k = 0; k < 4; ++k) {
        float2 p[4], q[4];  // units 2k, 2k+1 of the rows, then 2k+8, 2k+9; the same of the columns
#pragma unroll
        for (int i = 0; i < 4; ++i) p[i] = f2(__shfl_sync(FULL, a[i], (lane & 28) + k));
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            q[e] = f2(__shfl_sync(FULL, b.x, 8 * (lane & 3) + 4 * e + k));
            q[2 + e] = f2(__shfl_sync(FULL, b.y, 8 * (lane & 3) + 4 * e + k));
        }
#pragma unroll
        for (int r = 0; r < 2; ++r)
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                float &s = c[2 * r + e];
                s = fmaf(p[r].x, q[e].x, s);
                s = fmaf(p[r].y, q[e].y, s);
                s = fmaf(p[2 + r].x, q[2 + e].x, s);
                s = fmaf(p[2 + r].y, q[2 + e].y, s);
            }
    }
}
template <bool SIMT>
__device__ __forceinline__ void dot16(float (&c)[4], const unsigned (&a)[4], uint2 b) {
    if constexpr (SIMT) fma16(c, a, b);
    else mma16(c, a, b);
}
// Operand fragment of the 16 rows from `row`.
__device__ __forceinline__ void load_rows16(const uint2 *P16, int row, unsigned (&a)[4]) {
    const int lane = threadIdx.x & 31;
    const uint2 lo = P16[(size_t)(row + (lane >> 2)) * 4 + (lane & 3)];
    const uint2 hi = P16[(size_t)(row + 8 + (lane >> 2)) * 4 + (lane & 3)];
    a[0] = lo.x;
    a[1] = hi.x;
    a[2] = lo.y;
    a[3] = hi.y;
}
__device__ __forceinline__ uint2 load_cols8(const uint2 *P16, int col) {
    const int lane = threadIdx.x & 31;
    return P16[(size_t)(col + (lane >> 2)) * 4 + (lane & 3)];
}

// Packed FP32 pairs: two lanes of arithmetic per instruction, each rounded as
// its scalar counterpart.
__device__ __forceinline__ unsigned long long pack2(float lo, float hi) {
    unsigned long long r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ void unpack2(unsigned long long v, float &lo, float &hi) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ unsigned long long fma2(unsigned long long a, unsigned long long b, unsigned long long c) {
    unsigned long long r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ unsigned long long add2(unsigned long long a, unsigned long long b) {
    unsigned long long r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}

// Out of line: keeps the union-find loops out of the tile's registers.
static __device__ __noinline__ int unite_sets(int *parent, int x, int y, unsigned *status) {
    return db::uf_unite_root(parent, x, y, status);
}

// The state of one work item's 32 rows.  Lane l holds rows l/4 + 8 i, i < 4,
// of columns 2 (l mod 4) and the next in every group of 8.
template <int PASS, bool SIMT>
struct Item {
    unsigned a[2][4];             // operand fragments
    float an[4];                  // T + 1 - |p|^2, or -1e30 for a row the pass has no use for
    unsigned long long cnt[4];    // count: neighbours, even and odd columns apart
    int root[4];                  // merge: a member of each row's set
    int best[4];                  // border
    int was[2], now[2];           // merge: members lately joined, and a root found for each
    int row0;

    // Scores one column tile (64 columns from col0).
    __device__ __forceinline__ void tile(const Rows &R, int col0, int mytag, int ctag) {
        const int lane = threadIdx.x & 31;
        const float *nbcol = (PASS == WT_COUNT ? R.nb : R.nbc) + col0 + 2 * (lane & 3);
        const unsigned long long two = pack2(2.f, 2.f);
        unsigned any = 0;
#pragma unroll
        for (int h = 0; h < 2; ++h) {  // 32 columns: eight independent loads, then the scores
            uint2 b[4];
            float2 bn[4];
#pragma unroll
            for (int g = 0; g < 4; ++g) {
                b[g] = load_cols8(R.P16, col0 + 32 * h + 8 * g);
                bn[g] = *reinterpret_cast<const float2 *>(nbcol + 32 * h + 8 * g);
            }
#pragma unroll
            for (int g = 0; g < 4; ++g) {
                const unsigned long long q2 = pack2(bn[g].x, bn[g].y);
                unsigned hit = 0;  // bit 2 i + e: row i, column e
#pragma unroll
                for (int m = 0; m < 2; ++m) {
                    float c[4];
                    dot16<SIMT>(c, a[m], b[g]);
#pragma unroll
                    for (int k = 0; k < 2; ++k) {
                        const int i = 2 * m + k;
                        float w0, w1;  // 2 G - |q|^2
                        unpack2(fma2(pack2(c[2 * k], c[2 * k + 1]), two, q2), w0, w1);
                        if constexpr (PASS == WT_COUNT) {  // the score is an integer: saturated, 0 or 1
                            cnt[i] = add2(cnt[i], pack2(__saturatef(w0 + an[i]), __saturatef(w1 + an[i])));
                        } else {
                            hit |= (unsigned)(w0 + an[i] >= 1.f) << (2 * i);
                            hit |= (unsigned)(w1 + an[i] >= 1.f) << (2 * i + 1);
                        }
                    }
                }
                if constexpr (PASS == WT_COUNT) continue;
                if ((PASS == WT_NEAR || PASS == WT_FAR) && mytag >= 0 && ctag >= 0) {
                    any |= hit;
                    continue;
                }
                if (!__any_sync(FULL, hit)) continue;
                const int col = col0 + 32 * h + 8 * g + 2 * (lane & 3);
                if constexpr (PASS == WT_BORDER) {
                    if (hit) {
                        const int2 pt = *reinterpret_cast<const int2 *>(R.perm + col);
#pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            if ((hit >> (2 * i)) & 1u) best[i] = min(best[i], pt.x);
                            if ((hit >> (2 * i + 1)) & 1u) best[i] = min(best[i], pt.y);
                        }
                    }
                } else {
                    // members of the columns' sets; equal members need no union
                    int hq0 = 0, hq1 = 0;
                    if (hit) {
                        hq0 = member(db::ld_relaxed(R.parent + col));
                        hq1 = member(db::ld_relaxed(R.parent + col + 1));
                    }
                    for (; hit; hit &= hit - 1) {
                        const int bit = __ffs(hit) - 1, i = bit >> 1, e = bit & 1;
                        const int old = i < 2 ? (i ? root[1] : root[0]) : (i == 2 ? root[2] : root[3]);
                        const int hq = e ? hq1 : hq0;
                        if (hq == old) continue;
                        const int r = unite_sets(R.parent, old, hq, R.status);
#pragma unroll
                        for (int k = 0; k < 4; ++k)
                            if (root[k] == old || root[k] == hq) root[k] = r;
                        was[1] = was[0];
                        now[1] = now[0];
                        was[0] = hq;
                        now[0] = r;
                        if (hq0 == old || hq0 == hq) hq0 = r;
                        if (hq1 == old || hq1 == hq) hq1 = r;
                    }
                }
            }
        }
        // both tiles' core rows are one set each: one hit joins them
        if ((PASS == WT_NEAR || PASS == WT_FAR) && __any_sync(FULL, any) && lane == 0)
            unite_sets(R.parent, mytag, ctag, R.status);
    }

    // A row's parent, or the root that was found for it: rows not flattened since
    // the join would each ask for the same union again, two chained loads from
    // global memory at a time.
    __device__ __forceinline__ int member(int p) const { return p == was[0] ? now[0] : (p == was[1] ? now[1] : p); }

    // Neighbours counted so far of row i of this lane (the same in its quad).
    __device__ __forceinline__ int counted(int i) const {
        float lo, hi;
        unpack2(cnt[i], lo, hi);
        int v = (int)lo + (int)hi;
        v += __shfl_xor_sync(FULL, v, 1);
        v += __shfl_xor_sync(FULL, v, 2);
        return v;
    }
};

// Squared gap of two tiles' boxes (integers below 2^24 in FP32: exact).
__device__ __forceinline__ float box_gap2(const Rows &R, int s, int t, int d) {
    float gap2 = 0.f;
    for (int k = 0; k < d; ++k) {
        const float *lo = R.box + (size_t)k * R.cap_tiles, *hi = R.box + (size_t)(16 + k) * R.cap_tiles;
        const float g = fmaxf(fmaxf(lo[t] - hi[s], lo[s] - hi[t]), 0.f);
        gap2 = fmaf(g, g, gap2);
    }
    return gap2;
}

// One work item: rows [64 T + 32 half, + 32) against column tiles [ct0, ct1) of
// the batch.  Called by whole warps.
template <int PASS, bool SIMT>
__device__ __forceinline__ void run_item(const Rows &R, const TileRec &I, int T, int half, int ct0, int ct1) {
    const int lane = threadIdx.x & 31;
    const int mytag = PASS == WT_COUNT ? kMixed : R.tag[T];
    if ((PASS == WT_NEAR || PASS == WT_FAR) && mytag == kNoCore) return;
    if (PASS == WT_BORDER && !R.need[T]) return;
    const int left = I.n - ((T - I.tile0) * BT + 32 * half);  // rows of the instance from this half on
    if (left <= 0) return;
    Item<PASS, SIMT> it;
    it.row0 = T * BT + 32 * half;
    load_rows16(R.P16, it.row0, it.a[0]);
    load_rows16(R.P16, it.row0 + 16, it.a[1]);
    it.was[0] = it.was[1] = -3;  // no row
    it.now[0] = it.now[1] = -3;
    int prior[4];
    bool mine = false;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int row = it.row0 + (lane >> 2) + 8 * i;
        float b;
        if (PASS == WT_COUNT) b = R.nb[row];
        else if (PASS == WT_BORDER) b = !R.core[row] && R.count[row] > 1 ? R.nb[row] : -1e30f;  // exact: never left early
        else b = R.nbc[row];
        mine |= b > -1e29f;
        it.an[i] = I.Tp1 + b;
        it.cnt[i] = 0ull;
        it.best[i] = DB_NONE;
        it.root[i] = (PASS == WT_NEAR || PASS == WT_FAR) && b > -1e29f ? db::ld_relaxed(R.parent + row) : -2;
        prior[i] = PASS == WT_COUNT ? (b > -1e29f ? R.count[row] : INT_MAX / 2) : 0;
    }
    if (!__any_sync(FULL, mine)) return;
    if (PASS == WT_COUNT) {  // other chunks' items may have counted enough already
        bool done = true;
#pragma unroll
        for (int i = 0; i < 4; ++i) done &= prior[i] >= I.leave;
        if (__all_sync(FULL, done)) return;
    }
    unsigned long long evaluated = 0;
    const int rows_in = min(32, left), last = I.tile0 + I.ntiles - 1, nlast = I.n - (I.ntiles - 1) * BT;
    int visited = 0;
    auto visit = [&](int ct) {  // false: the rows are done
        it.tile(R, ct * BT, mytag, PASS == WT_NEAR || PASS == WT_FAR ? R.tag[ct] : 0);
        evaluated += (unsigned)(rows_in * (ct == last ? nlast : BT));
        ++visited;
        if (PASS != WT_COUNT || (visited > 2 && (visited & 1))) return true;
        bool done = true;
#pragma unroll
        for (int i = 0; i < 4; ++i) done &= prior[i] + it.counted(i) >= I.leave;
        return !__all_sync(FULL, done);
    };
    const int nct = ct1 - ct0, ngrp = (nct + 31) >> 5;
    const bool own = T >= ct0 && T < ct1;
    const int g0 = own ? (T - ct0) >> 5 : 0;
    bool more = true;
    for (int gi = 0; gi < ngrp && more; ++gi) {
        int g = g0 + gi;
        if (g >= ngrp) g -= ngrp;
        const int ct = ct0 + 32 * g + lane;
        bool in = ct < ct1 && box_gap2(R, T, ct, I.d) <= (float)I.Tc;
        if (PASS != WT_COUNT && in) {
            const int t = R.tag[ct];
            in = t != kNoCore;
            if (PASS == WT_FAR && in && t >= 0 && mytag >= 0)
                in = t != mytag && db::uf_find(R.parent, t) != db::uf_find(R.parent, mytag);
        }
        const unsigned m = __ballot_sync(FULL, in);
        // from the rows' own tile on, then the ones before it
        const int o = own && gi == 0 ? (T - ct0) & 31 : 0;
        unsigned hi = m & (FULL << o), lo = m & ~(FULL << o);
        for (; hi && more; hi &= hi - 1) more = visit(ct0 + 32 * g + __ffs(hi) - 1);
        for (; lo && more; lo &= lo - 1) more = visit(ct0 + 32 * g + __ffs(lo) - 1);
    }
    if (lane == 0 && R.ev && evaluated)
        atomicAdd(R.ev + 3 * I.inst + (PASS == WT_COUNT ? 0 : (PASS == WT_BORDER ? 2 : 1)), evaluated);
    if (PASS == WT_COUNT) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int v = it.counted(i), row = it.row0 + (lane >> 2) + 8 * i;
            if ((lane & 3) == 0 && (lane >> 2) + 8 * i < rows_in && v) atomicAdd(R.count + row, v);
        }
    }
    if (PASS == WT_BORDER) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            int v = it.best[i];
            v = min(v, __shfl_xor_sync(FULL, v, 1));
            v = min(v, __shfl_xor_sync(FULL, v, 2));
            if ((lane & 3) == 0 && v != DB_NONE) atomicMin(R.border + it.row0 + (lane >> 2) + 8 * i, v);
        }
    }
}

// Core flags of tile T, its core rows joined among themselves (each row's
// neighbours in the tile as a 64-bit mask, then smallest-label propagation in
// shared memory: no global atomics), and what follows: the masked norms, the
// tile's tag and whether some row needs the border pass.  A warp per tile, two
// rows a lane; adj and lab are the warp's own.
template <bool SIMT>
__device__ __forceinline__ void core_tile(const Rows &R, const TileRec &I, int T, unsigned long long *adj, int *lab) {
    const int lane = threadIdx.x & 31, r0 = (T - I.tile0) * BT;
    bool is[2], need[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int r = 32 * h + lane, row = T * BT + r;
        const int c = r0 + r < I.n ? R.count[row] : 0;
        is[h] = r0 + r < I.n && c >= I.min_pts;
        need[h] = !is[h] && c > 1;
        R.core[row] = is[h];
        R.border[row] = DB_NONE;
        R.nbc[row] = is[h] ? R.nb[row] : -1e30f;
        lab[r] = r;
    }
    const unsigned c0 = __ballot_sync(FULL, is[0]), c1 = __ballot_sync(FULL, is[1]);
    const int ncore = __popc(c0) + __popc(c1);
    const bool anyneed = __any_sync(FULL, need[0] || need[1]);
    int roots = ncore;
    if (ncore > 1) {
        // the 64 x 64 scores; lane l holds rows l/4 + 8 i of columns 2 (l mod 4) + e in each group of 8
        unsigned word[8][2];
        unsigned a[4][4];
        float an[8];
#pragma unroll
        for (int m = 0; m < 4; ++m) load_rows16(R.P16, T * BT + 16 * m, a[m]);
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int r = (lane >> 2) + 8 * i;
            const bool on = ((r < 32 ? c0 >> r : c1 >> (r - 32)) & 1u) != 0;
            an[i] = on ? I.Tp1 + R.nb[T * BT + r] : -1e30f;
            word[i][0] = word[i][1] = 0u;
        }
#pragma unroll
        for (int g = 0; g < 8; ++g) {
            const uint2 b = load_cols8(R.P16, T * BT + 8 * g);
            const int col = 8 * g + 2 * (lane & 3);
            const unsigned on = (col < 32 ? c0 >> col : c1 >> (col - 32)) & 3u;
            const float2 nb = *reinterpret_cast<const float2 *>(R.nb + T * BT + col);
            const float b0 = on & 1u ? nb.x : -1e30f, b1 = on & 2u ? nb.y : -1e30f;
#pragma unroll
            for (int m = 0; m < 4; ++m) {
                float c[4];
                dot16<SIMT>(c, a[m], b);
#pragma unroll
                for (int k = 0; k < 2; ++k) {
                    const unsigned e0 = fmaf(2.f, c[2 * k], b0) + an[2 * m + k] >= 1.f;
                    const unsigned e1 = fmaf(2.f, c[2 * k + 1], b1) + an[2 * m + k] >= 1.f;
                    word[2 * m + k][g >> 2] |= (e0 | (e1 << 1)) << (8 * (g & 3) + 2 * (lane & 3));
                }
            }
        }
#pragma unroll
        for (int i = 0; i < 8; ++i) {
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                word[i][h] |= __shfl_xor_sync(FULL, word[i][h], 1);
                word[i][h] |= __shfl_xor_sync(FULL, word[i][h], 2);
            }
            if ((lane & 3) == 0) adj[(lane >> 2) + 8 * i] = ((unsigned long long)word[i][1] << 32) | word[i][0];
        }
        __syncwarp();
        if (lane == 0 && R.ev) atomicAdd(R.ev + 3 * I.inst + 1, (unsigned long long)ncore * (ncore - 1) / 2);
        // every row under its smallest neighbour, flattened; then smaller labels
        // of any neighbour until none is left (a dense tile is one group at once)
        unsigned long long mask[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            mask[h] = is[h] ? adj[32 * h + lane] : 0ull;  // a core row is its own neighbour
            if (mask[h]) lab[32 * h + lane] = __ffsll((long long)mask[h]) - 1;
        }
        __syncwarp();
        while (true) {
            int l[2], least[2];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                l[h] = 32 * h + lane;
                while (lab[l[h]] < l[h]) l[h] = lab[l[h]];  // labels point to smaller rows
            }
            __syncwarp();
#pragma unroll
            for (int h = 0; h < 2; ++h) lab[32 * h + lane] = l[h];
            __syncwarp();
            roots = __popc(__ballot_sync(FULL, mask[0] && l[0] == lane)) +
                    __popc(__ballot_sync(FULL, mask[1] && l[1] == 32 + lane));
            if (roots <= 1) break;
            bool moved = false;
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                least[h] = l[h];
                for (unsigned long long m = mask[h]; m; m &= m - 1) least[h] = min(least[h], lab[__ffsll((long long)m) - 1]);
                moved |= least[h] < l[h];
            }
            if (!__any_sync(FULL, moved)) break;
#pragma unroll
            for (int h = 0; h < 2; ++h)
                if (least[h] < l[h]) {
                    atomicMin(&lab[l[h]], least[h]);  // the group's first row, too
                    atomicMin(&lab[32 * h + lane], least[h]);
                }
            __syncwarp();
        }
    }
    __syncwarp();
#pragma unroll
    for (int h = 0; h < 2; ++h) R.parent[T * BT + 32 * h + lane] = T * BT + lab[32 * h + lane];
    if (lane == 0) {
        const int first = c0 ? __ffs(c0) - 1 : 32 + __ffs(c1) - 1;  // the first core row
        R.tag[T] = ncore == 0 ? kNoCore : (roots == 1 ? T * BT + first : kMixed);
        R.need[T] = anyneed;
    }
    __syncwarp();
}

// Every core row of a tile straight under its root, and the tile's tag (left
// as it is when the tile has no core row): a warp per tile, two rows a lane.
__device__ __forceinline__ void flatten_tile(const Rows &R, int T) {
    const int lane = threadIdx.x & 31;
    int lo = INT_MAX, hi = -1;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int row = T * BT + 32 * h + lane;
        if (R.core[row]) {
            const int root = db::uf_find(R.parent, row);
            if (root != row) db::st_relaxed(R.parent + row, root);
            lo = min(lo, root);
            hi = max(hi, root);
        }
    }
    lo = __reduce_min_sync(FULL, lo);
    hi = __reduce_max_sync(FULL, hi);
    if (lane == 0 && hi >= 0) R.tag[T] = lo == hi ? lo : kMixed;
}

// Root of a core row, and the smallest point index of each set: one atomic per
// distinct root of the warp, and none that cannot lower the value.  Every lane
// of the warp calls it.
__device__ __forceinline__ void root_row(int *parent, int *least, bool is, int row, int point) {
    const int lane = threadIdx.x & 31;
    const int root = is ? db::uf_settle(parent, row) : -1 - lane;
    const unsigned peers = __match_any_sync(FULL, root);
    if (is) {
        const int m = __reduce_min_sync(peers, point);
        if (lane == __ffs(peers) - 1 && m < db::ld_relaxed(least + root)) atomicMin(least + root, m);
    }
}

// ---- the passes, as kernels ----

// Work item w: half w mod 2 of tile T of some step, with the chunk `step` after
// the tile's own (wrapping around its instance), for one warp; the next item is
// claimed while the current one runs.  TABLE: first holds the tiles before each
// step (batch_items.h); else all tiles have max_chunks chunks.
template <int PASS, bool TABLE, bool SIMT>
static __global__ void __launch_bounds__(NT, 3) pass_kernel(Rows R, const Hdr *__restrict__ hdr, int ch_tiles,
                                                     const unsigned *__restrict__ first, unsigned *work) {
    db::wait_prior_grid();  // returns at once when launched the plain way
    db::allow_next_grid();
    const int lane = threadIdx.x & 31;
    const unsigned total = (unsigned)hdr->total_tiles, steps = PASS == WT_NEAR ? 1u : (unsigned)hdr->max_chunks;
    const unsigned nitems = 2u * (TABLE && PASS != WT_NEAR ? first[steps] : total * steps);
    int step = 0;
    unsigned next = 0;
    if (lane == 0) next = atomicAdd(work, 1u);
    while (true) {
        const unsigned item = __shfl_sync(FULL, next, 0);
        if (item >= nitems) return;
        if (lane == 0) next = atomicAdd(work, 1u);
        if (TABLE && PASS != WT_NEAR) step = batchitems::step_at(item >> 1, step, first);
        else step = (int)((item >> 1) / total);
        const int T = (int)((item >> 1) - (TABLE && PASS != WT_NEAR ? first[step] : (unsigned)step * total));
        const TileRec I = R.tiles[T];
        const int end = I.tile0 + I.ntiles;
        int ct0, ct1;
        if (PASS == WT_NEAR) {
            ct0 = T + 1;
            ct1 = min(end, T + 1 + kNear);
        } else {
            const int nchunk = (I.ntiles + ch_tiles - 1) / ch_tiles;
            int chunk = (T - I.tile0) / ch_tiles + step;
            if (chunk >= nchunk) chunk -= nchunk;
            ct0 = I.tile0 + chunk * ch_tiles;
            ct1 = min(end, ct0 + ch_tiles);
            if (PASS == WT_FAR) ct0 = max(ct0, T + 1 + kNear);
        }
        if (ct0 < ct1) run_item<PASS, SIMT>(R, I, T, (int)(item & 1), ct0, ct1);
    }
}

template <bool SIMT>
static __global__ void __launch_bounds__(NT, 3) core_kernel(Rows R, const Hdr *__restrict__ hdr) {
    db::wait_prior_grid();
    db::allow_next_grid();
    __shared__ unsigned long long adj[NT / 32][BT];
    __shared__ int lab[NT / 32][BT];
    const int total = hdr->total_tiles, nwarps = (int)((gridDim.x * blockDim.x) >> 5), wib = threadIdx.x >> 5;
    for (int T = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5); T < total; T += nwarps)
        core_tile<SIMT>(R, R.tiles[T], T, adj[wib], lab[wib]);
}

static __global__ void __launch_bounds__(NT) flatten_kernel(Rows R, const Hdr *__restrict__ hdr) {
    db::wait_prior_grid();
    db::allow_next_grid();
    const int total = hdr->total_tiles, nwarps = (int)((gridDim.x * blockDim.x) >> 5);
    for (int T = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5); T < total; T += nwarps) flatten_tile(R, T);
}

static __global__ void __launch_bounds__(NT) root_kernel(Rows R, const Hdr *__restrict__ hdr, int *least) {
    db::wait_prior_grid();
    db::allow_next_grid();
    const int total = hdr->total_tiles * BT, step = (int)(gridDim.x * blockDim.x);
    for (int g0 = (int)(blockIdx.x * blockDim.x); g0 < total; g0 += step) {
        const int g = g0 + (int)threadIdx.x;
        const bool is = g < total && R.core[g];
        root_row(R.parent, least, is, g, is ? R.perm[g] : 0);
    }
}

// ---- packing ----

// What packing writes, by row, tile or point (see Rows).
struct PackOut {
    TileRec *tiles;
    int *perm, *inv, *count, *least;
    uint2 *P16;
    float *nb, *box;
    long long cap_tiles;
};

__device__ __forceinline__ unsigned half2_bits(int lo, int hi) {
    const __half2 h = __halves2half2(__int2half_rn(lo), __int2half_rn(hi));
    return *reinterpret_cast<const unsigned *>(&h);
}

// Packs the 64 rows of tile tt of an instance (a warp, two rows a lane): grid
// check, centred units, norm, the tile's box.  A lane reads its two rows whole
// (the rows of a tile are scattered in the input), all loads independent.
// order: point of each row (null: identity).  Returns true on off-grid input.
template <int DP, typename Order>
__device__ __forceinline__ bool pack_tile(const float *x, const TileRec &I, int tt, const Order *order,
                                          const PackOut &w) {
    const int lane = threadIdx.x & 31, n = I.n, d = I.d, T = I.tile0 + tt;
    bool bad = false;
    int v[2][DP];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int s = tt * BT + 32 * h + lane, row = T * BT + 32 * h + lane;
        const int o = s < n ? (order ? (int)order[s] : s) : 0;
        const float *src = x + (size_t)o * d;
        float f[DP];
#pragma unroll
        for (int k = 0; k < DP; ++k) f[k] = s < n && k < d ? src[k] : 0.5f;
        if (s < n) {
            w.perm[row] = o;
            w.inv[I.point0 + o] = row;
        }
        w.count[row] = 0;
        w.least[row] = DB_NONE;
        int s2 = 0;
#pragma unroll
        for (int k = 0; k < DP; ++k) {
            int u;
            bad |= !db::on_grid(f[k], u);
            v[h][k] = u - 512;  // 0 for the padding
            s2 += v[h][k] * v[h][k];
        }
        w.nb[row] = s < n ? -(float)s2 : -1e30f;
#pragma unroll
        for (int k = 0; k < 4; ++k) {  // piece k: units 2k, 2k+1, 2k+8, 2k+9
            uint2 pc;
            pc.x = half2_bits(2 * k < DP ? v[h][2 * k] : 0, 2 * k + 1 < DP ? v[h][2 * k + 1] : 0);
            pc.y = half2_bits(2 * k + 8 < DP ? v[h][2 * k + 8] : 0, 2 * k + 9 < DP ? v[h][2 * k + 9] : 0);
            w.P16[(size_t)row * 4 + k] = pc;
        }
    }
    const bool on0 = tt * BT + lane < n, on1 = tt * BT + 32 + lane < n;
#pragma unroll
    for (int k = 0; k < DP; ++k) {
        const int lo = __reduce_min_sync(FULL, min(on0 ? v[0][k] : INT_MAX, on1 ? v[1][k] : INT_MAX));
        const int hi = __reduce_max_sync(FULL, max(on0 ? v[0][k] : INT_MIN, on1 ? v[1][k] : INT_MIN));
        if (lane == 0) {
            w.box[(size_t)k * w.cap_tiles + T] = (float)lo;
            w.box[(size_t)(16 + k) * w.cap_tiles + T] = (float)hi;
        }
    }
    if (lane == 0) w.tiles[T] = I;
    return bad;
}
template <typename Order>
__device__ __forceinline__ bool pack_tile_d(const float *x, const TileRec &I, int tt, const Order *order,
                                            const PackOut &w) {
    switch (I.d) {  // warp-uniform
        case 1: return pack_tile<1>(x, I, tt, order, w);
        case 2: return pack_tile<2>(x, I, tt, order, w);
        case 3: return pack_tile<3>(x, I, tt, order, w);
        case 4: return pack_tile<4>(x, I, tt, order, w);
        case 5:
        case 6:
        case 7:
        case 8: return pack_tile<8>(x, I, tt, order, w);
        default: return pack_tile<16>(x, I, tt, order, w);
    }
}

// Morton (Z-order) dilation of a 10-bit coordinate: bit b moves to bit 3b.
__device__ __forceinline__ unsigned dilate3(unsigned v) {
    v &= 1023u;
    v = (v | (v << 16)) & 0x030000FFu;
    v = (v | (v << 8)) & 0x0300F00Fu;
    v = (v | (v << 4)) & 0x030C30C3u;
    v = (v | (v << 2)) & 0x09249249u;
    return v;
}

// Z-order code of a point's first dz (at most three) grid coordinates, the top
// `bits` bits of each interleaved.
__device__ __forceinline__ unsigned zcode(const float *x, int dz, int bits) {
    unsigned code = 0;
    for (int j = 0; j < dz; ++j) {
        int u;
        db::on_grid(x[j], u);  // off-grid input is reported when the row is packed
        code |= dilate3((unsigned)u >> (10 - bits)) << j;
    }
    if (dz == 3) return code;
    unsigned c = 0;  // no third (second) axis: close the gaps
    for (int b = 0; b < bits; ++b) c |= ((code >> (3 * b)) & ((1u << dz) - 1u)) << (dz * b);
    return c;
}

}  // namespace wtile
