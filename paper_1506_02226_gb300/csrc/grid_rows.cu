// grid_rows.cu — the eps-grid path for d <= 3 with cells in key order.
//
// Geometry, exact test and labels are grid.cu's.  There the cells are numbered
// in the order in which blocks find them, so a cell's neighbours lie anywhere
// and each is looked up by itself (up to 124 table lookups a cell, 89 of 402 us
// for 500,000 points in space) and listed.  Here cell ids follow the cell keys
// (x fastest), and points are grouped in that order: the occupied cells of a
// run of neighbouring cells along x are consecutive ids and their points one
// contiguous range.  A cell's neighbourhood is then at most 5 (plane) or 25
// (space) ranges, found by two rank lookups each, and empty rows cost nothing
// more.
//
// Rank of a key (occupied cells before it), two forms:
//   direct   when all G^d cells fit the cell table: counts per key, one scan of
//            cells and points gives idx[key] and the ranges;
//   bitmap   otherwise, when one bit per cell fits its buffer: per 32 cells the
//            bits and the occupied cells before them (a scan of the words);
//            points are then counted per id and scanned.
// Larger grids (eps tiny against the data's extent) take grid.cu, and so do more
// than kMaxN points: the most that these kernels have been run with.  They are
// the faster ones there too (400 groups plus 20% noise, this file / grid.cu:
// 1,048,576 points 350 / 510 us in the plane and 640 / 1,070 in space, 4,194,304
// points 453 / 672 us and 3.87 / 6.01 ms).
//
// Kernels: prep, scans (2 kernels direct, 5 with the bitmap), scatter beside
// rows (the range lists), count, border beside the merge, roots, labels.  The
// merge's forest is over cells, linked towards smaller ids:
//   hook     every cell with cores under the first neighbouring cell before it
//            whose central core point is within eps of its own: plain stores, no
//            search.  Only cells with no such neighbour stay roots, a few at the
//            lower rim of each group (under the neighbour with the smallest
//            representative, every local minimum of the representatives stayed
//            one, and the union took 138 us for 500,000 points in space);
//   flatten  every cell straight under its root;
//   union    cell pairs whose roots still differ: central points, then, when the
//            cells hold few pairs, all of them, a lane per cell pair; most cell
//            pairs are skipped by one comparison;
//   search   what is left, a list, a warp per cell pair (searched where they
//            were found, a cell with a score of them held up its warp: the merge
//            of 500,000 points in space took 141 us instead of 97).
#include <algorithm>
#include <climits>
#include <type_traits>
#include <cmath>

#include "grid_dev.cuh"

namespace {

constexpr int64_t kMaxN = int64_t(1) << 22;
constexpr int kWalkThreads = 64; // count and border blocks: a warp next to a tight blob holds up few others
constexpr int kLaneTests = 64;   // merge: pairs of two cells that a single lane tests
constexpr int kScanTile = 2048;  // entries per block of a scan: 256 threads x 8

struct RowGeom {
    int d, c, G, nrows;  // nrows: rows of neighbouring cells along x, the own row in two parts
    float Tp1, inv_c;
    int ncells_all;      // G^d (bitmap: below 2^31)
    // {oy, oz, reach along x, kind}: kind 0 a whole row, 1 the own row left of the cell, 2 right of it
    char4 row[26];
};

struct RowArgs {
    RowGeom g;
    int n;
    const unsigned long long *ctr0;  // (cells << 32) | points
    const uint2 *rk;          // bitmap: {occupied cells before the word, its bits}
    const int *idx;           // direct: occupied cells before each key
    const unsigned *cell_at;  // by id: cell coordinates cx | cy << 10 | cz << 20
    int *start;               // first position of each cell's points, [cells + 1]
    int4 *rows;               // {first id, end id, first position, end position}, stride g.nrows
    int *nent, *cand;         // entries of a cell's list, points in them
    const float4 *spts;
    const int *sidx, *scell;
    uint8_t *score;
    int *rep;                 // smallest core index of each cell
    unsigned long long *mid;  // (squared distance to the centre << 32) | packed point
    int *par;                 // forest of cells
    int *least;               // smallest representative of each set, at its root
    int *bord;
    int2 *pairs;              // merge: cell pairs left to a warp each, and their number
    int *npairs, pair_cap;
    unsigned *status, *status_out;
    unsigned long long *ev;   // pair tests: [0] count, [1] merge, [2] border
};

// Cell coordinates of a key (the divisions are made once per cell).
__device__ __forceinline__ unsigned cell_of_key(unsigned key, int G) {
    const unsigned row = key / (unsigned)G, cx = key - row * (unsigned)G, cz = row / (unsigned)G, cy = row - cz * (unsigned)G;
    return cx | (cy << 10) | (cz << 20);
}

__device__ __forceinline__ unsigned key_of_point(const int *u, const RowGeom &g) {
    const unsigned cx = (unsigned)(u[0] / g.c), cy = g.d > 1 ? (unsigned)(u[1] / g.c) : 0u,
                   cz = g.d > 2 ? (unsigned)(u[2] / g.c) : 0u;
    return (cz * (unsigned)g.G + cy) * (unsigned)g.G + cx;
}

// Grid check and cell key of every point.  Direct: counts per key, and the
// point's place among them, with one atomic per distinct cell of the warp.
// Bitmap: the cell's bit, set once.
template <bool DIRECT>
__global__ void __launch_bounds__(256) rows_prep_kernel(const float *__restrict__ x, int n, RowGeom g, int *cnt,
                                                        unsigned *bits, unsigned *__restrict__ key_out,
                                                        int *__restrict__ rank, float4 *__restrict__ pts4,
                                                        unsigned *status) {
    db::wait_prior_grid();  // started as a programmatic dependent
    db::allow_next_grid();
    const int i = blockIdx.x * blockDim.x + threadIdx.x, lane = threadIdx.x & 31;
    const bool valid = i < n;
    unsigned key = 0;
    if (valid) {
        int u[3] = {0, 0, 0};
        bool ok = true;
        for (int k = 0; k < g.d; ++k) ok &= db::on_grid(x[(size_t)i * g.d + k], u[k]);
        if (!ok) atomicOr(status, DB_EBIT_NOT_QUANTISED);
        key = key_of_point(u, g);
        const float f0 = (float)u[0], f1 = (float)u[1], f2 = (float)u[2];
        pts4[i] = make_float4(f0, f1, f2, -(f0 * f0 + f1 * f1 + f2 * f2));
        key_out[i] = key;
    }
    const unsigned peers = __match_any_sync(FULL, valid ? key : 0x80000000u + lane);  // keys are below 2^31
    const int leader = __ffs(peers) - 1;
    if (DIRECT) {
        int base = 0;
        if (valid && lane == leader) base = atomicAdd(cnt + key, __popc(peers));
        base = __shfl_sync(FULL, base, leader);
        if (valid) rank[i] = base + __popc(peers & db::lanemask_lt());
    } else if (valid && lane == leader) {
        const unsigned b = 1u << (key & 31u);
        if (!((unsigned)db::ld_relaxed(reinterpret_cast<const int *>(bits) + (key >> 5)) & b)) atomicOr(bits + (key >> 5), b);
    }
}

// ---- scans: block totals, then every block adds up the totals before it ----

// What an entry contributes: DIRECT (occupied, points) of a key, WORDS occupied
// cells of a bitmap word, COUNTS the points of a cell.
enum { SCAN_DIRECT = 0, SCAN_WORDS = 1, SCAN_COUNTS = 2 };

template <int WHAT>
__device__ __forceinline__ unsigned long long scan_value(unsigned v) {
    if (WHAT == SCAN_DIRECT) return ((unsigned long long)(v != 0u) << 32) | v;
    if (WHAT == SCAN_WORDS) return (unsigned long long)__popc(v) << 32;
    return v;
}

struct ScanArgs {
    const unsigned *in;
    int m;                     // entries (COUNTS: at most; the cells are on the device)
    unsigned long long *part;  // block totals
    unsigned long long *ctr0;
    int n;
    uint2 *rk;
    int *idx;
    unsigned *cell_at;
    int *start;
    int G;
};

template <int WHAT>
__device__ __forceinline__ unsigned long long load8(const ScanArgs &a, int i0, int m, unsigned (&v)[8]) {
    unsigned long long s = 0;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        v[k] = i0 + k < m ? a.in[i0 + k] : 0u;
        s += scan_value<WHAT>(v[k]);
    }
    return s;
}

__device__ __forceinline__ unsigned long long block_sum_u64(unsigned long long v, unsigned long long *red) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(FULL, v, o);
    __syncthreads();
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    __syncthreads();
    unsigned long long t = 0;
#pragma unroll
    for (int w = 0; w < 8; ++w) t += red[w];
    return t;
}

template <int WHAT>
__global__ void __launch_bounds__(256) rows_sums_kernel(ScanArgs a) {
    db::wait_prior_grid();
    db::allow_next_grid();
    __shared__ unsigned long long red[8];
    const int m = WHAT == SCAN_COUNTS ? (int)(*a.ctr0 >> 32) : a.m;
    unsigned v[8];
    const unsigned long long t = block_sum_u64(load8<WHAT>(a, blockIdx.x * kScanTile + threadIdx.x * 8, m, v), red);
    if (threadIdx.x == 0) a.part[blockIdx.x] = t;
}

template <int WHAT>
__global__ void __launch_bounds__(256) rows_apply_kernel(ScanArgs a) {
    db::wait_prior_grid();
    db::allow_next_grid();
    __shared__ unsigned long long red[8], wt[8];
    const int t = threadIdx.x, lane = t & 31, wid = t >> 5;
    const int m = WHAT == SCAN_COUNTS ? (int)(*a.ctr0 >> 32) : a.m;
    unsigned long long before = 0;  // totals of the blocks before this one
    for (int b = t; b < (int)blockIdx.x; b += 256) before += a.part[b];
    before = block_sum_u64(before, red);
    const int i0 = blockIdx.x * kScanTile + t * 8;
    unsigned v[8];
    const unsigned long long s = load8<WHAT>(a, i0, m, v);
    unsigned long long inc = s;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned long long y = __shfl_up_sync(FULL, inc, o);
        if (lane >= o) inc += y;
    }
    if (lane == 31) wt[wid] = inc;
    __syncthreads();
    unsigned long long at = before + inc - s;
#pragma unroll
    for (int w = 0; w < 8; ++w)
        if (w < wid) at += wt[w];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        const int i = i0 + k;
        if (i < m) {
            const int id = (int)(at >> 32), first = (int)(at & 0xffffffffull);
            if (WHAT == SCAN_DIRECT) {
                a.idx[i] = id;
                if (v[k]) {
                    a.cell_at[id] = cell_of_key((unsigned)i, a.G);
                    a.start[id] = first;
                }
            } else if (WHAT == SCAN_WORDS) {
                a.rk[i] = make_uint2((unsigned)id, v[k]);
            } else {
                a.start[i] = first;
            }
            at += scan_value<WHAT>(v[k]);
            if (i == m - 1) {  // the last entry: what the whole scan adds up to
                if (WHAT == SCAN_DIRECT) a.idx[m] = (int)(at >> 32);
                if (WHAT != SCAN_COUNTS) *a.ctr0 = ((at >> 32) << 32) | (unsigned)a.n;
                if (WHAT != SCAN_WORDS) a.start[WHAT == SCAN_DIRECT ? (int)(at >> 32) : m] = a.n;
            }
        }
    }
}

// Occupied cells before `key`.
template <bool DIRECT>
__device__ __forceinline__ int cells_before(const RowArgs &a, unsigned key) {
    if (DIRECT) return a.idx[key];
    const uint2 w = a.rk[key >> 5];
    return (int)(w.x + __popc(w.y & ((1u << (key & 31u)) - 1u)));
}

// Bitmap: the id of every point's cell, points per cell and the point's place
// among them (one atomic per distinct cell of the warp).
__global__ void __launch_bounds__(256) rows_cellcount_kernel(RowArgs a, unsigned *__restrict__ key_io,
                                                             unsigned *__restrict__ cell_at, int *cnt,
                                                             int *__restrict__ rank) {
    db::wait_prior_grid();
    db::allow_next_grid();
    const int i = blockIdx.x * blockDim.x + threadIdx.x, lane = threadIdx.x & 31;
    const bool valid = i < a.n;
    const unsigned key = valid ? key_io[i] : 0u;
    const int id = valid ? cells_before<false>(a, key) : -1 - lane;
    const unsigned peers = __match_any_sync(FULL, id);
    const int leader = __ffs(peers) - 1;
    int base = 0;
    if (valid && lane == leader) {
        base = atomicAdd(cnt + id, __popc(peers));
        if (base == 0) cell_at[id] = cell_of_key(key, a.g.G);
    }
    base = __shfl_sync(FULL, base, leader);
    if (!valid) return;
    rank[i] = base + __popc(peers & db::lanemask_lt());
    key_io[i] = (unsigned)id;
}

template <bool DIRECT>
__global__ void __launch_bounds__(256) rows_scatter_kernel(RowArgs a, const unsigned *__restrict__ key,
                                                           const int *__restrict__ rank,
                                                           const float4 *__restrict__ pts4, float4 *__restrict__ spts,
                                                           int *__restrict__ sidx, int *__restrict__ scell) {
    db::wait_prior_grid();
    db::allow_next_grid();
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= a.n) return;
    const int id = DIRECT ? a.idx[key[i]] : (int)key[i];
    const int pos = a.start[id] + rank[i];
    spts[pos] = pts4[i];
    sidx[pos] = i;
    scell[pos] = id;
}

// Range lists, RL lanes per cell, a lane per row of neighbouring cells.
template <bool DIRECT, int RL>
__global__ void __launch_bounds__(256) rows_list_kernel(RowArgs a) {
    db::wait_prior_grid();
    db::allow_next_grid();
    __shared__ char4 srow[32];
    if (threadIdx.x < 32) srow[threadIdx.x] = threadIdx.x < a.g.nrows ? a.g.row[threadIdx.x] : make_char4(0, 0, 0, -1);
    __syncthreads();
    const int lane = threadIdx.x & 31, r = lane & (RL - 1), grp = lane & ~(RL - 1);
    const int ncells = (int)(*a.ctr0 >> 32), G = a.g.G;
    const char4 o = srow[r];
    const int step = (int)(gridDim.x * blockDim.x) / RL;
    // two cells per round: their lookups are independent chains
    for (int c0 = (int)(blockIdx.x * blockDim.x + threadIdx.x - r) / RL; c0 - grp / RL < ncells; c0 += 2 * step) {
        int4 e[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int c = c0 + h * step;
            e[h] = make_int4(0, 0, 0, 0);
            if (c < ncells && r < a.g.nrows) {
                const unsigned at = a.cell_at[c];
                const int cx = (int)(at & 1023u), cy = (int)((at >> 10) & 1023u), cz = (int)(at >> 20);
                const int y = cy + o.x, z = cz + o.y;
                if (y >= 0 && y < G && z >= 0 && z < G) {
                    const unsigned row = ((unsigned)z * (unsigned)G + (unsigned)y) * (unsigned)G;
                    const int lo = max(0, cx - o.z), hi = min(G - 1, cx + o.z);
                    e[h].x = o.w == 2 ? c + 1 : cells_before<DIRECT>(a, row + lo);
                    e[h].y = o.w == 1 ? c : cells_before<DIRECT>(a, row + hi + 1);
                }
            }
        }
#pragma unroll
        for (int h = 0; h < 2; ++h)
            if (e[h].x < e[h].y) {
                e[h].z = a.start[e[h].x];
                e[h].w = a.start[e[h].y];
            }
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int c = c0 + h * step;
            const bool on = e[h].x < e[h].y;
            const unsigned m = (__ballot_sync(FULL, on) >> grp) & (RL == 32 ? FULL : ((1u << (RL & 31)) - 1u));
            if (on) a.rows[(size_t)c * a.g.nrows + __popc(m & ((1u << r) - 1u))] = e[h];
            int t = e[h].w - e[h].z;
#pragma unroll
            for (int k = RL / 2; k > 0; k >>= 1) t += __shfl_xor_sync(FULL, t, k);
            if (c < ncells) {
                if (r == 0) {
                    a.nent[c] = __popc(m);
                    a.cand[c] = t;
                    a.rep[c] = DB_NONE;
                }
                if (r == 1) {  // and the first state of the later passes
                    a.mid[c] = ~0ull;
                    a.par[c] = c;
                    a.least[c] = DB_NONE;
                }
            }
        }
    }
}

// Count pass (Section IV-B, fused pair test + count), a thread per grouped
// position.  The points of its own cell are neighbours (a clique); the others
// lie in the ranges of its cell's list, which the thread walks itself when they
// hold few points and together with the warp's other points of that cell, 128
// candidates a step, when they hold many.  Otherwise as in grid.cu.
template <int D>
__global__ void __launch_bounds__(kWalkThreads) rows_count_kernel(RowArgs a, int min_pts, int exact, int *counts_out,
                                                         uint8_t *core_out) {
    db::wait_prior_grid();
    db::allow_next_grid();
    const int lane = threadIdx.x & 31, p = blockIdx.x * blockDim.x + threadIdx.x;
    const bool valid = p < a.n;
    const int lim = exact ? INT_MAX : min_pts;
    const int A = valid ? a.scell[p] : -1 - lane;  // no two invalid lanes share a cell
    unsigned long long ev = 0;
    int cnt = 0, o = DB_NONE;
    bool heavy = false;
    float4 pt = make_float4(0.f, 0.f, 0.f, 0.f);
    if (valid) {
        cnt = a.start[A + 1] - a.start[A];
        pt = a.spts[p];
        o = a.sidx[p];
    }
    const float cp = a.g.Tp1 + pt.w, px2 = 2.f * pt.x, py2 = 2.f * pt.y, pz2 = 2.f * pt.z;
    if (valid && cnt < lim) {
        heavy = a.cand[A] > kThreadWalkMax;
        if (!heavy) {
            const int4 *row = a.rows + (size_t)A * a.g.nrows;
            const int ne = a.nent[A];
            for (int k0 = 0; k0 < ne && cnt < lim; k0 += 4) {
                int s[4], e[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const int4 en = k0 + u < ne ? row[k0 + u] : make_int4(0, 0, 0, 0);
                    s[u] = en.z;
                    e[u] = en.w;
                }
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    ev += (unsigned)(e[u] - s[u]);
#pragma unroll 4
                    for (int q = s[u]; q < e[u]; ++q) cnt += is_nbr<D>(cp, px2, py2, pz2, a.spts[q]);
                }
            }
        }
    }
    unsigned hv = __ballot_sync(FULL, heavy);
    while (hv) {
        const int H = __shfl_sync(FULL, A, __ffs(hv) - 1);
        const unsigned mine = __ballot_sync(FULL, heavy && A == H);
        hv &= ~mine;
        const int ne = a.nent[H];
        unsigned pend = mine;
        const int4 en = lane < ne ? a.rows[(size_t)H * a.g.nrows + lane] : make_int4(0, 0, 0, 0);  // at most 26
        const int s = en.z, c = en.w - en.z;
        const int incl = warp_incl_scan(c), total = __shfl_sync(FULL, incl, 31);
        for (int base = 0; base < total && pend; base += 128) {
            float4 qq[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int j = base + 32 * u + lane, k = locate_lane(j, incl);
                const int ex = __shfl_sync(FULL, incl, k) - __shfl_sync(FULL, c, k);  // lane k's first j
                const int q = __shfl_sync(FULL, s, k) + (j - ex);
                qq[u] = j < total ? a.spts[q] : make_float4(0.f, 0.f, 0.f, -1e30f);
            }
            if (lane == 0) ev += (unsigned long long)__popc(pend) * (unsigned)min(128, total - base);
            for (unsigned m = pend; m; m &= m - 1) {
                const int i = __ffs(m) - 1;
                const float cpi = __shfl_sync(FULL, cp, i), px2i = __shfl_sync(FULL, px2, i);
                const float py2i = D > 1 ? __shfl_sync(FULL, py2, i) : 0.f, pz2i = D > 2 ? __shfl_sync(FULL, pz2, i) : 0.f;
                int add = 0;
#pragma unroll
                for (int u = 0; u < 4; ++u) add += is_nbr<D>(cpi, px2i, py2i, pz2i, qq[u]);
                const int r = (int)__reduce_add_sync(FULL, (unsigned)add);
                if (lane == i) cnt += r;
            }
            pend = __ballot_sync(FULL, ((mine >> lane) & 1u) && cnt < lim);
        }
    }
    if (valid) {
        const bool core = cnt >= min_pts;
        a.score[p] = core;
        if (counts_out) counts_out[o] = cnt;
        if (core_out) core_out[o] = core;
        if (!core) o = DB_NONE;
    }
    // the core point nearest A's centre, in doubled grid units
    unsigned long long mid = ~0ull;
    if (o != DB_NONE) {
        const int c = a.g.c, ux = (int)pt.x, uy = (int)pt.y, uz = (int)pt.z;
        const int dx = 2 * ux - (2 * (int)((pt.x + 0.5f) * a.g.inv_c) * c + c - 1);
        const int dy = D > 1 ? 2 * uy - (2 * (int)((pt.y + 0.5f) * a.g.inv_c) * c + c - 1) : 0;
        const int dz = D > 2 ? 2 * uz - (2 * (int)((pt.z + 0.5f) * a.g.inv_c) * c + c - 1) : 0;
        mid = ((unsigned long long)(unsigned)(dx * dx + dy * dy + dz * dz) << 32) |
              (unsigned)(ux | (uy << 10) | (uz << 20));
    }
    o = seg_min_down(o, A);
    mid = seg_min_down(mid, A);
    const int Aprev = __shfl_up_sync(FULL, A, 1);
    if (valid && (lane == 0 || Aprev != A) && o != DB_NONE) {
        atomicMin(a.rep + A, o);
        atomicMin(a.mid + A, mid);
    }
    db::block_sum_add(a.ev + 0, ev);
}

// ---- merge (Section IV-C) ----

template <int D, int RL>
__global__ void __launch_bounds__(256) rows_hook_kernel(RowArgs a) {
    db::wait_prior_grid();
    db::allow_next_grid();
    const int lane = threadIdx.x & 31, r = lane & (RL - 1), grp = lane & ~(RL - 1);
    const int ncells = (int)(*a.ctr0 >> 32), step = (int)(gridDim.x * blockDim.x) / RL;
    unsigned long long ev = 0;
    for (int c0 = (int)(blockIdx.x * blockDim.x + threadIdx.x - r) / RL; c0 - grp / RL < ncells; c0 += step) {
        const int c = c0;
        const int repc = c < ncells ? a.rep[c] : DB_NONE;
        if (!__any_sync(FULL, repc != DB_NONE)) continue;
        int best = INT_MAX;
        if (repc != DB_NONE && r < a.nent[c]) {
            const int4 e = a.rows[(size_t)c * a.g.nrows + r];
            const int end = min(e.y, c);
            const float4 m = unpack_point(a.mid[c]);
            const float cp = a.g.Tp1 + m.w, mx2 = 2.f * m.x, my2 = 2.f * m.y, mz2 = 2.f * m.z;
            unsigned long long mq[5];  // a row holds at most five cells; no core point: all ones
#pragma unroll
            for (int k = 0; k < 5; ++k) mq[k] = e.x + k < end ? a.mid[e.x + k] : ~0ull;
#pragma unroll
            for (int k = 4; k >= 0; --k)
                if (mq[k] != ~0ull) {
                    ++ev;
                    if (is_nbr<D>(cp, mx2, my2, mz2, unpack_point(mq[k]))) best = e.x + k;
                }
        }
        if (RL == 32) {
            best = __reduce_min_sync(FULL, best);
        } else {
#pragma unroll
            for (int k = RL / 2; k > 0; k >>= 1) best = min(best, __shfl_xor_sync(FULL, best, k));
        }
        if (r == 0 && best != INT_MAX) a.par[c] = best;
    }
    db::block_sum_add(a.ev + 1, ev);
}

__global__ void __launch_bounds__(256) rows_flatten_kernel(RowArgs a) {
    db::wait_prior_grid();
    db::allow_next_grid();
    const int ncells = (int)(*a.ctr0 >> 32);
    for (int c = (int)(blockIdx.x * blockDim.x + threadIdx.x); c < ncells; c += (int)(gridDim.x * blockDim.x)) {
        const int root = db::uf_find(a.par, c);
        if (root != c) db::st_relaxed(a.par + c, root);
    }
}

template <int D, int RL>
__global__ void __launch_bounds__(256) rows_union_kernel(RowArgs a) {
    db::wait_prior_grid();
    db::allow_next_grid();
    const int lane = threadIdx.x & 31, r = lane & (RL - 1), grp = lane & ~(RL - 1);
    const int ncells = (int)(*a.ctr0 >> 32), step = (int)(gridDim.x * blockDim.x) / RL;
    unsigned long long ev = 0;
    for (int c0 = (int)(blockIdx.x * blockDim.x + threadIdx.x - r) / RL; c0 - grp / RL < ncells; c0 += step) {
        const int c = c0;
        const int repc = c < ncells ? a.rep[c] : DB_NONE;
        if (!__any_sync(FULL, repc != DB_NONE)) continue;
        int4 e = make_int4(0, 0, 0, 0);
        int root = -1;
        if (repc != DB_NONE && r < a.nent[c]) {
            e = a.rows[(size_t)c * a.g.nrows + r];
            e.x = max(e.x, c + 1);  // each cell pair from its smaller id
            root = db::ld_relaxed(a.par + c);
        }
        // roots as the flattening left them: equal ones are one set (sets only
        // merge); a row holds at most five cells, looked at together
        unsigned differ = 0;
#pragma unroll
        for (int k = 0; k < 5; ++k)
            if (e.x + k < e.y)
                differ |= (unsigned)(a.rep[e.x + k] != DB_NONE && db::ld_relaxed(a.par + e.x + k) != root) << k;
        while (__any_sync(FULL, differ)) {
            const int id = e.x + (differ ? __ffs((int)differ) - 1 : 0);
            bool need = differ != 0;
            differ &= differ - 1;
            if (need) need = db::uf_find(a.par, c) != db::uf_find(a.par, id);
            if (need) {  // the two central core points first, lanes in parallel
                const float4 m = unpack_point(a.mid[c]);
                ++ev;
                bool hit = is_nbr<D>(a.g.Tp1 + m.w, 2.f * m.x, 2.f * m.y, 2.f * m.z, unpack_point(a.mid[id]));
                const int sA = a.start[c], eA = a.start[c + 1], sB = a.start[id], eB = a.start[id + 1];
                // few pairs (64 bits: two hot spots make more than an int holds): the lane tests them itself
                if (!hit && (long long)(eA - sA) * (eB - sB) <= kLaneTests) {
                    need = false;
                    for (int qa = sA; qa < eA && !hit; ++qa) {
                        if (!a.score[qa]) continue;
                        const float4 pa = a.spts[qa];
                        const float cp = a.g.Tp1 + pa.w, px2 = 2.f * pa.x, py2 = 2.f * pa.y, pz2 = 2.f * pa.z;
#pragma unroll 4
                        for (int qb = sB; qb < eB; ++qb) {
                            const bool t = a.score[qb];
                            ev += t;
                            hit |= t && is_nbr<D>(cp, px2, py2, pz2, a.spts[qb]);
                        }
                    }
                }
                if (hit) {
                    db::uf_unite(a.par, c, id, a.status);
                    need = false;
                }
            }
            const unsigned left = __ballot_sync(FULL, need);  // many pairs: a warp each, in the next kernel
            if (left) {
                int base = 0;
                if (lane == __ffs(left) - 1) base = atomicAdd(a.npairs, __popc(left));
                base = __shfl_sync(FULL, base, __ffs(left) - 1) + __popc(left & db::lanemask_lt());
                // (the list holds two pairs a point; what it cannot take the lane searches)
                if (need && base < a.pair_cap) {
                    a.pairs[base] = make_int2(c, id);
                } else if (need) {
                    bool hit = false;
                    for (int qa = a.start[c]; qa < a.start[c + 1] && !hit; ++qa)
                        for (int qb = a.start[id]; qb < a.start[id + 1] && !hit && a.score[qa]; ++qb) {
                            const float4 pa = a.spts[qa];
                            hit = a.score[qb] &&
                                  is_nbr<D>(a.g.Tp1 + pa.w, 2.f * pa.x, 2.f * pa.y, 2.f * pa.z, a.spts[qb]);
                        }
                    if (hit) db::uf_unite(a.par, c, id, a.status);
                }
            }
        }
    }
    db::block_sum_add(a.ev + 1, ev);
}

// The listed cell pairs, a warp each: 128 points of the smaller cell staged at
// a time, the lanes over the larger one.
template <int D>
__global__ void __launch_bounds__(256) rows_search_kernel(RowArgs a) {
    db::wait_prior_grid();
    db::allow_next_grid();
    __shared__ float4 ybuf[8][128];
    __shared__ uint8_t ycore[8][128];
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    const int npairs = min(*a.npairs, a.pair_cap), nwarps = (int)((gridDim.x * blockDim.x) >> 5);
    float4 *yb = ybuf[wib];
    uint8_t *yc = ycore[wib];
    unsigned long long ev = 0;
    for (int k = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5); k < npairs; k += nwarps) {
        const int2 pr = a.pairs[k];
        const int A = pr.x, B = pr.y;
        const int sA = a.start[A], cA = a.start[A + 1] - sA, sB = a.start[B], cB = a.start[B + 1] - sB;
        int same = 0;
        if (lane == 0) same = db::uf_find(a.par, A) == db::uf_find(a.par, B);
        if (__shfl_sync(FULL, same, 0)) continue;
        const bool swap = cB > cA;  // lanes over the larger cell
        const int sX = swap ? sB : sA, cX = swap ? cB : cA, sY = swap ? sA : sB, cY = swap ? cA : cB;
        bool found = false;
        for (int y0 = 0; y0 < cY && !found; y0 += 128) {
            const int ny = min(128, cY - y0);
            __syncwarp();
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int q = lane + 32 * u;
                if (q < ny) {
                    yb[q] = a.spts[sY + y0 + q];
                    yc[q] = a.score[sY + y0 + q];
                }
            }
            __syncwarp();
            for (int x0 = 0; x0 < cX && !found; x0 += 32) {
                const int xi = x0 + lane;
                const bool vx = xi < cX && a.score[sX + xi];
                const unsigned vxm = __ballot_sync(FULL, vx);
                if (!vxm) continue;
                const float4 px = a.spts[sX + (xi < cX ? xi : 0)];
                const float cp = a.g.Tp1 + px.w, px2 = 2.f * px.x, py2 = 2.f * px.y, pz2 = 2.f * px.z;
                for (int q = 0; q < ny; ++q) {
                    if (!yc[q]) continue;
                    if (lane == 0) ev += (unsigned)__popc(vxm);
                    if (__any_sync(FULL, vx && is_nbr<D>(cp, px2, py2, pz2, yb[q]))) {
                        found = true;
                        break;
                    }
                }
            }
        }
        if (found && lane == 0) db::uf_unite(a.par, A, B, a.status);
        __syncwarp();
    }
    db::block_sum_add(a.ev + 1, ev);
}

// Border pass: each non-core point takes its smallest-index core neighbour, a
// thread per grouped position, with the count's split of the walks; bord[p]
// gets the cell of the chosen core point (DB_NONE for noise).
template <int D>
__global__ void __launch_bounds__(kWalkThreads) rows_border_kernel(RowArgs a) {
    db::wait_prior_grid();
    db::allow_next_grid();
    const int lane = threadIdx.x & 31, p = blockIdx.x * blockDim.x + threadIdx.x;
    const bool valid = p < a.n, mine = valid && !a.score[p];
    const int A = valid ? a.scell[p] : -1 - lane;
    unsigned long long ev = 0;
    int best = DB_NONE, bc = DB_NONE;
    bool heavy = false;
    float4 pt = make_float4(0.f, 0.f, 0.f, 0.f);
    if (mine) {
        best = a.rep[A];
        bc = best != DB_NONE ? A : DB_NONE;
        pt = a.spts[p];
        heavy = a.cand[A] > kThreadWalkMax;
    }
    const float cp = a.g.Tp1 + pt.w, px2 = 2.f * pt.x, py2 = 2.f * pt.y, pz2 = 2.f * pt.z;
    if (mine && !heavy) {
        const int4 *row = a.rows + (size_t)A * a.g.nrows;
        const int ne = a.nent[A];
        for (int k0 = 0; k0 < ne; k0 += 4) {
            int s[4], e[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int4 en = k0 + u < ne ? row[k0 + u] : make_int4(0, 0, 0, 0);
                s[u] = en.z;
                e[u] = en.w;
            }
#pragma unroll
            for (int u = 0; u < 4; ++u)
#pragma unroll 4
                for (int q = s[u]; q < e[u]; ++q) {
                    const uint8_t sc = a.score[q];  // independent loads
                    const int qi = a.sidx[q];
                    const float4 pq = a.spts[q];
                    if (sc && qi < best) {
                        ++ev;
                        if (is_nbr<D>(cp, px2, py2, pz2, pq)) {
                            best = qi;
                            bc = a.scell[q];
                        }
                    }
                }
        }
    }
    unsigned hv = __ballot_sync(FULL, heavy);
    while (hv) {
        const int H = __shfl_sync(FULL, A, __ffs(hv) - 1);
        const unsigned mineH = __ballot_sync(FULL, heavy && A == H);
        hv &= ~mineH;
        const int4 en = lane < a.nent[H] ? a.rows[(size_t)H * a.g.nrows + lane] : make_int4(0, 0, 0, 0);
        const int s = en.z, c = en.w - en.z;
        const int incl = warp_incl_scan(c), total = __shfl_sync(FULL, incl, 31);
        for (int base = 0; base < total; base += 128) {
            float4 qq[4];
            int qi[4], qc[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int j = base + 32 * u + lane, k = locate_lane(j, incl);
                const int ex = __shfl_sync(FULL, incl, k) - __shfl_sync(FULL, c, k);  // lane k's first j
                const int q = __shfl_sync(FULL, s, k) + (j - ex);
                const bool v = j < total;
                const uint8_t scq = v ? a.score[q] : 0;  // independent loads
                const int qv = v ? a.sidx[q] : DB_NONE;
                qq[u] = v ? a.spts[q] : make_float4(0.f, 0.f, 0.f, -1e30f);
                qc[u] = v ? a.scell[q] : 0;
                qi[u] = scq ? qv : DB_NONE;
            }
            for (unsigned m = mineH; m; m &= m - 1) {
                const int i = __ffs(m) - 1;
                const int bi = __shfl_sync(FULL, best, i);
                bool any = false;
#pragma unroll
                for (int u = 0; u < 4; ++u) any |= qi[u] < bi;
                if (!__any_sync(FULL, any)) continue;  // no core index of these can beat the current best
                const float cpi = __shfl_sync(FULL, cp, i), px2i = __shfl_sync(FULL, px2, i);
                const float py2i = D > 1 ? __shfl_sync(FULL, py2, i) : 0.f, pz2i = D > 2 ? __shfl_sync(FULL, pz2, i) : 0.f;
                int lb = bi, lc = DB_NONE;
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const bool better = qi[u] < lb;  // else the pair needs no test
                    ev += better;
                    if (better && is_nbr<D>(cpi, px2i, py2i, pz2i, qq[u])) {
                        lb = qi[u];
                        lc = qc[u];
                    }
                }
                const int nb = (int)__reduce_min_sync(FULL, (unsigned)lb);
                if (nb < bi) {  // warp-uniform: the one lane holding nb has its cell
                    const int w = __ffs(__ballot_sync(FULL, lb == nb)) - 1;
                    const int cw = __shfl_sync(FULL, lc, w);
                    if (lane == i) {
                        best = nb;
                        bc = cw;
                    }
                }
            }
        }
    }
    if (mine) a.bord[p] = bc;
    db::block_sum_add(a.ev + 2, ev);
}

// Root of every cell with cores, and the smallest representative of each set.
__global__ void __launch_bounds__(256) rows_root_kernel(RowArgs a) {
    db::wait_prior_grid();
    db::allow_next_grid();
    const int ncells = (int)(*a.ctr0 >> 32), step = (int)(gridDim.x * blockDim.x), lane = threadIdx.x & 31;
    for (int c0 = (int)(blockIdx.x * blockDim.x); c0 < ncells; c0 += step) {
        const int c = c0 + (int)threadIdx.x, rep = c < ncells ? a.rep[c] : DB_NONE;
        const int root = rep != DB_NONE ? db::uf_settle(a.par, c) : -1 - lane;
        // one atomic per distinct root of the warp, and none that cannot lower the value
        const unsigned peers = __match_any_sync(FULL, root);
        if (rep != DB_NONE) {
            const int m = __reduce_min_sync(peers, rep);
            if (lane == __ffs(peers) - 1 && m < db::ld_relaxed(a.least + root)) atomicMin(a.least + root, m);
        }
    }
}

// Labels, a thread per grouped point: the label of its cell's set (core) or of
// the set of its chosen core neighbour's cell (border), noise -1; and the
// statistics (a cluster's label is the index of one of its core points).
__global__ void __launch_bounds__(256) rows_label_kernel(RowArgs a, int *__restrict__ labels, unsigned long long *ctr) {
    db::wait_prior_grid();
    db::allow_next_grid();
    db::report_status(a.status, a.status_out);
    __shared__ int red[4];
    if (threadIdx.x < 4) red[threadIdx.x] = 0;
    __syncthreads();
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    int kind = -1;
    bool root = false;
    if (p < a.n) {
        const int o = a.sidx[p];
        const bool core = a.score[p];
        const int c = core ? a.scell[p] : a.bord[p];
        int lab = -1;
        kind = core ? 0 : (c == DB_NONE ? 2 : 1);
        if (kind != 2) lab = a.least[a.par[c]];
        root = core && lab == o;
        labels[o] = lab;
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const unsigned m = __ballot_sync(FULL, k < 3 ? kind == k : root);
        if ((threadIdx.x & 31) == 0 && m) atomicAdd(&red[k], __popc(m));
    }
    __syncthreads();
    if (threadIdx.x < 4 && red[threadIdx.x]) atomicAdd(ctr + 2 + threadIdx.x, (unsigned long long)red[threadIdx.x]);
}

// Ordered candidate pairs: every cell's points times the points of its
// neighbourhood, itself included.
__global__ void __launch_bounds__(256) rows_candidates_kernel(RowArgs a, unsigned long long *out) {
    const int ncells = (int)(*a.ctr0 >> 32);
    unsigned long long s = 0;
    for (int c = (int)(blockIdx.x * blockDim.x + threadIdx.x); c < ncells; c += (int)(gridDim.x * blockDim.x)) {
        const unsigned long long m = (unsigned)(a.start[c + 1] - a.start[c]);
        s += m * (m + (unsigned)a.cand[c]);
    }
    db::block_sum_add(out, s);
}

// Rows of neighbouring cells along x from g's kept offsets: an offset set is
// symmetric and holds every |ox| up to a row's reach.
RowGeom row_geometry(const GridGeom &g) {
    RowGeom r{};
    r.d = g.d;
    r.c = g.c;
    r.G = g.G;
    r.Tp1 = g.Tp1;
    r.inv_c = g.inv_c;
    r.ncells_all = 1;
    for (int k = 0; k < g.d; ++k) r.ncells_all *= g.G;
    int reach[5][5];
    for (auto &y : reach)
        for (int &z : y) z = -1;
    reach[2][2] = 0;
    for (int k = 0; k < g.noff; ++k) {
        int &w = reach[g.off[k].y + 2][g.off[k].z + 2];
        w = std::max(w, std::abs((int)g.off[k].x));
    }
    r.row[r.nrows++] = make_char4(0, 0, (signed char)reach[2][2], 1);
    r.row[r.nrows++] = make_char4(0, 0, (signed char)reach[2][2], 2);
    for (int ring = 1; ring <= 2; ++ring)  // near rows first
        for (int z = -2; z <= 2; ++z)
            for (int y = -2; y <= 2; ++y)
                if (std::max(std::abs(y), std::abs(z)) == ring && reach[y + 2][z + 2] >= 0)
                    r.row[r.nrows++] = make_char4((signed char)y, (signed char)z, (signed char)reach[y + 2][z + 2], 0);
    return r;
}

cudaStream_t fork(const DbWork &w, cudaStream_t st, int k) {
    if (!w.side || w.marks->on) return st;
    cudaEventRecord(w.fj[k], st);
    cudaStreamWaitEvent(w.side, w.fj[k], 0);
    return w.side;
}

void join(const DbWork &w, cudaStream_t st, cudaStream_t s2, int k) {
    if (s2 == st) return;
    cudaEventRecord(w.fj[k], s2);
    cudaStreamWaitEvent(st, w.fj[k], 0);
}

template <bool DIRECT, int D>
cudaError_t run_rows(const DbWork &w, const RowGeom &g, const float *x, int n, int min_pts, bool exact, bool stats,
                     int32_t *labels, int32_t *counts_out, uint8_t *core_out, cudaStream_t st) {
    constexpr int RL = D == 3 ? 32 : 8;  // lanes per cell: at least its rows (2, 6, 26)
    unsigned *key = reinterpret_cast<unsigned *>(w.slot_of);
    int *rank = w.count, *start = w.scan, *cnt = w.hcount;
    unsigned long long *mid = reinterpret_cast<unsigned long long *>(w.cell_mid);  // 8 of its 16 bytes per cell
    RowArgs a{};
    a.g = g;
    a.n = n;
    a.ctr0 = w.ctr;
    a.rk = w.rk;
    a.idx = reinterpret_cast<const int *>(w.hkey);
    a.cell_at = w.cell_key;
    a.start = start;
    a.rows = reinterpret_cast<int4 *>(w.nbr);
    a.nent = w.ncnt;
    a.cand = w.cell_cand;
    a.spts = w.spts;
    a.sidx = w.sidx;
    a.scell = w.scell;
    a.score = w.score;
    a.rep = w.cell_rep;
    a.mid = mid;
    a.par = w.cell_start;
    a.least = w.hcursor;
    a.bord = w.border;
    a.pairs = reinterpret_cast<int2 *>(w.pts4);  // free after the scatter: two pairs a point
    a.pair_cap = 2 * n;
    a.npairs = reinterpret_cast<int *>(w.ctr + DB_CTR_PAIRS);
    a.status = w.status;
    a.status_out = w.status_out;
    a.ev = w.ctr + DB_CTR_EVAL;
    ScanArgs s{};
    s.part = w.rg_part;
    s.ctr0 = w.ctr;
    s.n = n;
    s.rk = w.rk;
    s.idx = reinterpret_cast<int *>(w.hkey);
    s.cell_at = w.cell_key;
    s.start = start;
    s.G = g.G;
    const int nb = (n + 255) / 256;
    auto scan = [&](auto what, const unsigned *in, int m, const char *nm) {
        constexpr int WHAT = decltype(what)::value;
        s.in = in;
        s.m = m;
        const int blocks = (m + kScanTile - 1) / kScanTile;
        launch_dependent(rows_sums_kernel<WHAT>, blocks, 256, st, s);
        w.marks->kernel("grid_sums", st);
        launch_dependent(rows_apply_kernel<WHAT>, blocks, 256, st, s);
        w.marks->kernel(nm, st);
    };
    launch_dependent(rows_prep_kernel<DIRECT>, nb, 256, st, x, n, g, cnt, w.occ, key, rank, w.pts4, w.status);
    w.marks->kernel("grid_prep", st);
    if constexpr (DIRECT) {
        scan(std::integral_constant<int, SCAN_DIRECT>{}, reinterpret_cast<const unsigned *>(cnt), g.ncells_all, "grid_cells");
    } else {
        scan(std::integral_constant<int, SCAN_WORDS>{}, w.occ, g.ncells_all / 32 + 1, "grid_words");
        launch_dependent(rows_cellcount_kernel, nb, 256, st, a, key, w.cell_key, cnt, rank);
        w.marks->kernel("grid_cellcount", st);
        scan(std::integral_constant<int, SCAN_COUNTS>{}, reinterpret_cast<const unsigned *>(cnt), n, "grid_cells");
    }
    // the range lists need the cells but not the grouped points
    const int cgrid = (int)std::min<int64_t>(((int64_t)n * RL + 255) / 256, 152 * 8);
    cudaStream_t s2 = fork(w, st, 0);
    launch_dependent(rows_list_kernel<DIRECT, RL>, cgrid, 256, s2, a);
    w.marks->kernel("grid_rows", s2);
    launch_dependent(rows_scatter_kernel<DIRECT>, nb, 256, st, a, key, rank, w.pts4, w.spts, w.sidx, w.scell);
    w.marks->kernel("grid_scatter", st);
    join(w, st, s2, 1);
    launch_dependent(rows_count_kernel<D>, (n + kWalkThreads - 1) / kWalkThreads, kWalkThreads, st, a, min_pts, exact ? 1 : 0, counts_out, core_out);
    w.marks->kernel("grid_count", st);
    // the border pass needs the core flags but not the merge: it runs beside it
    s2 = fork(w, st, 2);
    launch_dependent(rows_border_kernel<D>, (n + kWalkThreads - 1) / kWalkThreads, kWalkThreads, s2, a);
    w.marks->kernel("grid_border", s2);
    launch_dependent(rows_hook_kernel<D, RL>, cgrid, 256, st, a);
    w.marks->kernel("grid_hook", st);
    launch_dependent(rows_flatten_kernel, std::min(nb, 152 * 8), 256, st, a);
    w.marks->kernel("grid_flatten", st);
    launch_dependent(rows_union_kernel<D, RL>, cgrid, 256, st, a);
    w.marks->kernel("grid_union_near", st);
    launch_dependent(rows_search_kernel<D>, std::min(nb, 152 * 6), 256, st, a);
    w.marks->kernel("grid_search", st);
    launch_dependent(rows_root_kernel, std::min(nb, 152 * 8), 256, st, a);
    w.marks->kernel("grid_root", st);
    join(w, st, s2, 3);
    launch_dependent(rows_label_kernel, nb, 256, st, a, labels, w.ctr);
    w.marks->kernel("grid_label", st);
    if (stats) {
        rows_candidates_kernel<<<152 * 4, 256, 0, st>>>(a, w.ctr + 1);
        w.marks->kernel("grid_candidates", st);
    }
    return cudaGetLastError();
}

}  // namespace

bool grid_rows_serves(const DbWork &w, const GridGeom &g, int64_t n) {
    int64_t all = 1;
    for (int k = 0; k < g.d; ++k) all *= g.G;
    return n <= kMaxN && w.rk && all < (int64_t(1) << 31) && (all < w.hcap || all / 32 + 1 <= w.occ_cap);
}

// Clears the counters itself, and the status word when `reset` is set.
cudaError_t launch_grid_rows(const DbWork &w, const GridGeom &g0, const float *x, int64_t n64, int32_t min_pts,
                             bool exact, bool stats, bool reset, int32_t *labels, int32_t *counts_out,
                             uint8_t *core_out, cudaStream_t st) {
    const int n = (int)n64;
    const RowGeom g = row_geometry(g0);
    const bool direct = g.ncells_all < w.hcap;
    // status, counters and counts lie one after the other
    char *from = reset ? reinterpret_cast<char *>(w.status) : reinterpret_cast<char *>(w.ctr);
    const size_t bytes = reinterpret_cast<char *>(w.hcount) - from + sizeof(int) * (size_t)(direct ? g.ncells_all : n);
    cudaError_t e;
    if ((e = cudaMemsetAsync(from, 0, bytes, st))) return e;
    if (!direct && (e = cudaMemsetAsync(w.occ, 0, sizeof(unsigned) * ((size_t)g.ncells_all / 32 + 1), st))) return e;
#define DB_ROWS(DIRECT)                                                                                              \
    (g.d == 1 ? run_rows<DIRECT, 1>(w, g, x, n, min_pts, exact, stats, labels, counts_out, core_out, st)             \
              : (g.d == 2 ? run_rows<DIRECT, 2>(w, g, x, n, min_pts, exact, stats, labels, counts_out, core_out, st) \
                          : run_rows<DIRECT, 3>(w, g, x, n, min_pts, exact, stats, labels, counts_out, core_out, st)))
    return direct ? DB_ROWS(true) : DB_ROWS(false);
#undef DB_ROWS
}
