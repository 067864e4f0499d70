// grid_small.cu — the eps-grid path for small point sets (d <= 3, up to 4,096
// points), in one launch.
//
// The grid path (grid.cu) is a chain of some ten kernels; with a few thousand
// points each of them works for a microsecond or two, and the launches, the
// clears and the gaps between them are what a call takes (2,000 points in the
// plane: 100 us).  Here one thread block cluster runs the whole method: every
// block bins all points into its own shared memory (the binning is cheaper than
// sharing it), counts neighbours and finds border neighbours for its eighth of
// the points, and takes its eighth of the cell pairs in the merge.  The blocks
// meet twice (cluster barriers): when the core flags are known (each block
// writes its points' flags into every block's shared memory) and when the
// merge, a union-find in global memory, is complete.
//
// The geometry, the exact test, the order of decisions and so the labels are
// grid.cu's: cells are cliques, cell pairs within the kept offsets are
// candidates, a cell's representative is its smallest core index, and only
// representatives are linked.
#include <cooperative_groups.h>

#include <climits>

#include "internal.cuh"

namespace cg = cooperative_groups;

namespace {

constexpr int kMaxN = kGridSmallMaxN;  // 4,096
constexpr int NB = 8, NT = 512;        // blocks of the cluster, threads of a block: at most one own point a thread
constexpr int kSlots = 2 * kMaxN;      // cell hash
constexpr int kList = 2048;            // merge: cell pairs left to a whole warp
constexpr int kThreadTests = 64;       // merge: pair tests a thread makes before it leaves a cell pair to a warp
constexpr unsigned FULL = 0xffffffffu;

struct SmallSmem {
    float4 pt[kMaxN];         // {u0, u1, u2, -|u|^2} grouped by cell
    unsigned key[kSlots];     // cell hash
    unsigned range[kSlots];   // (first position << 16) | points of the cell
    int rep[kSlots];          // smallest core index of the cell (first: fill cursor)
    unsigned list[kList];     // (slot << 16) | slot
    uint16_t cell[kMaxN];     // slots of the occupied cells
    uint16_t idx[kMaxN];      // point at each position
    uint16_t pos[kMaxN];      // position of each point; then this block's cells in the merge
    uint16_t slot[kMaxN];     // cell of each position
    uint8_t core[kMaxN];      // by point (written by all blocks)
    uint8_t score[kMaxN];     // by position
    char4 off[128];
    int wsum[NT / 32], wocc[NT / 32];
    unsigned bits[kMaxN / 32 + 1];  // roots, when labels are made dense
    int before[kMaxN / 32 + 1];
    int nlist, nown;
    int red[4];
};

struct SmallArgs {
    const float *x;
    int n, hbits, min_pts, exact, compact, stats, reset;
    GridGeom g;
    int *parent, *labels, *counts_out;
    uint8_t *core_out;
    unsigned *status;
    unsigned long long *ctr;
};

// Cluster barrier in two halves, each entered by converged warps (the aligned
// forms require it, and the per-point loops before them end at different times).
__device__ __forceinline__ void cluster_arrive() {
    __syncthreads();
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_wait() {
    __syncthreads();
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// Slot of a cell, -1 when it holds no point.
__device__ __forceinline__ int find_cell(const SmallSmem &S, unsigned key, int bits) {
    const unsigned mask = (1u << bits) - 1u;
    unsigned h = db::hash_slot(key, bits);
    for (unsigned probe = 0; probe <= mask; ++probe) {
        const unsigned k = S.key[h];
        if (k == key) return (int)h;
        if (k == DB_HASH_EMPTY) return -1;
        h = (h + 1) & mask;
    }
    return -1;
}

__device__ __forceinline__ unsigned key_of(int cx, int cy, int cz, int G) {
    return ((unsigned)cz * (unsigned)G + (unsigned)cy) * (unsigned)G + (unsigned)cx;
}

// Key of the cell at offset o from cell (cx, cy, cz); false outside the grid.
__device__ __forceinline__ bool key_at(int cx, int cy, int cz, char4 o, int G, unsigned &key) {
    const int x = cx + o.x, y = cy + o.y, z = cz + o.z;
    key = key_of(x, y, z, G);
    return x >= 0 && x < G && y >= 0 && y < G && z >= 0 && z < G;
}

// T + 1 - D(p,q) >= 1, exact (grid.cu).
__device__ __forceinline__ bool near(float cp, float px2, float py2, float pz2, float4 q) {
    return fmaf(pz2, q.z, fmaf(py2, q.y, fmaf(px2, q.x, cp + q.w))) >= 1.f;
}

__global__ void __cluster_dims__(NB, 1, 1) __launch_bounds__(NT, 1) grid_small_kernel(SmallArgs a) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    SmallSmem &S = *reinterpret_cast<SmallSmem *>(smem_raw);
    cg::cluster_group cluster = cg::this_cluster();
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5, rank = (int)cluster.block_rank();
    const int n = a.n, G = a.g.G, noff = a.g.noff, nslots = 1 << a.hbits, d = a.g.d;
    const float Tp1 = a.g.Tp1;
    // all blocks have started before any writes to another's shared memory
    cluster_arrive();

    // ---- every block bins all points ----
    for (int h = tid; h < nslots; h += NT) {
        S.key[h] = DB_HASH_EMPTY;
        S.range[h] = 0u;
    }
    if (tid < 128) S.off[tid] = tid < noff ? a.g.off[tid] : make_char4(0, 0, 0, 0);
    if (tid == 0) S.nlist = S.nown = 0;
    if (tid < 4) S.red[tid] = 0;
    if (rank == 0 && tid < DB_NCTR) a.ctr[tid] = 0ull;
    if (rank == 0 && tid == 0 && a.reset) *a.status = 0u;
    constexpr int PER = kMaxN / NT;
    float f[PER][3];
#pragma unroll
    for (int k = 0; k < PER; ++k) {
        const int i = tid + k * NT;
#pragma unroll
        for (int c = 0; c < 3; ++c) f[k][c] = i < n && c < d ? a.x[(size_t)i * d + c] : 0.f;
    }
    __syncthreads();
    bool ok = true;
    unsigned packed[PER];
    int slot[PER];
#pragma unroll
    for (int k = 0; k < PER; ++k) {
        const int i = tid + k * NT;
        slot[k] = -1;
        if (i >= n) continue;
        int u[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) ok &= db::on_grid(f[k][c], u[c]);
        packed[k] = (unsigned)u[0] | ((unsigned)u[1] << 10) | ((unsigned)u[2] << 20);
        const unsigned key = key_of(u[0] / a.g.c, u[1] / a.g.c, u[2] / a.g.c, G);
        unsigned h = db::hash_slot(key, a.hbits);
        for (int probe = 0; probe < nslots; ++probe) {  // at least 2 n slots: ends
            const unsigned cur = atomicCAS(&S.key[h], DB_HASH_EMPTY, key);
            if (cur == DB_HASH_EMPTY || cur == key) break;
            h = (h + 1) & (unsigned)(nslots - 1);
        }
        slot[k] = (int)h;
        atomicAdd(&S.range[h], 1u);
    }
    __syncthreads();
    // first positions and the list of occupied cells: each thread a run of slots
    const int per = nslots / NT;  // 2 to 16 (hbits >= 10)
    int cnt = 0, occ = 0;
    for (int k = 0; k < per; ++k) {
        const int c = (int)S.range[tid * per + k];
        cnt += c;
        occ += c > 0;
    }
    int ic = cnt, io = occ;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int yc = __shfl_up_sync(FULL, ic, o), yo = __shfl_up_sync(FULL, io, o);
        if (lane >= o) {
            ic += yc;
            io += yo;
        }
    }
    if (lane == 31) {
        S.wsum[wid] = ic;
        S.wocc[wid] = io;
    }
    __syncthreads();
    int at = ic - cnt, cid = io - occ, ncells = 0;
    for (int w = 0; w < NT / 32; ++w) {
        if (w < wid) {
            at += S.wsum[w];
            cid += S.wocc[w];
        }
        ncells += S.wocc[w];
    }
    for (int k = 0; k < per; ++k) {
        const int h = tid * per + k, c = (int)S.range[h];
        if (!c) continue;
        S.range[h] = ((unsigned)at << 16) | (unsigned)c;
        S.rep[h] = at;  // fill cursor
        S.cell[cid++] = (uint16_t)h;
        at += c;
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < PER; ++k) {
        if (slot[k] < 0) continue;
        const int p = atomicAdd(&S.rep[slot[k]], 1);
        const float x = (float)(packed[k] & 1023u), y = (float)((packed[k] >> 10) & 1023u), z = (float)(packed[k] >> 20);
        S.pt[p] = make_float4(x, y, z, -(x * x + y * y + z * z));
        S.idx[p] = (uint16_t)(tid + k * NT);
        S.pos[tid + k * NT] = (uint16_t)p;
        S.slot[p] = (uint16_t)slot[k];
    }
    __syncthreads();
    for (int c = tid; c < ncells; c += NT) S.rep[S.cell[c]] = DB_NONE;

    // ---- neighbour counts of this block's points ----
    const int own = (n + NB - 1) / NB, i = rank * own + tid;
    const bool mine = tid < own && i < n;
    float4 p = make_float4(0.f, 0.f, 0.f, 0.f);
    int A = 0, cx = 0, cy = 0, cz = 0, count = 0;
    unsigned long long ev_count = 0, ev_merge = 0, ev_border = 0, cand = 0;
    if (mine) {
        const int q = S.pos[i];
        p = S.pt[q];
        A = S.slot[q];
        const unsigned keyA = S.key[A];
        cx = (int)(keyA % (unsigned)G);
        cy = (int)((keyA / (unsigned)G) % (unsigned)G);
        cz = (int)(keyA / ((unsigned)G * (unsigned)G));
        count = (int)(S.range[A] & 0xffffu);  // the cell is a clique
        a.parent[i] = i;
    }
    const float cp = Tp1 + p.w, px2 = 2.f * p.x, py2 = 2.f * p.y, pz2 = 2.f * p.z;
    const int lim = a.exact ? INT_MAX : a.min_pts;
    if (mine) {
        cand = (unsigned)count;
        for (int o = 0; o < noff; ++o) {
            if (count >= lim && !a.stats) break;
            unsigned key;
            if (!key_at(cx, cy, cz, S.off[o], G, key)) continue;
            const int B = find_cell(S, key, a.hbits);
            if (B < 0) continue;
            const unsigned r = S.range[B];
            const int q0 = (int)(r >> 16), q1 = q0 + (int)(r & 0xffffu);
            cand += r & 0xffffu;
            if (count >= lim) continue;
            for (int q = q0; q < q1; ++q) count += near(cp, px2, py2, pz2, S.pt[q]);
            ev_count += r & 0xffffu;
        }
    }
    cluster_wait();
    if (mine)
        for (int r = 0; r < NB; ++r) cluster.map_shared_rank(S.core, r)[i] = count >= a.min_pts;
    cluster_arrive();
    cluster_wait();  // core flags, the forest's first state and the cleared counters are everywhere
    if (!ok) atomicOr(a.status, DB_EBIT_NOT_QUANTISED);

    // ---- representatives, by every block ----
    for (int q = tid; q < n; q += NT) {
        const int o = S.idx[q];
        const uint8_t c = S.core[o];
        S.score[q] = c;
        if (c) atomicMin(&S.rep[S.slot[q]], o);
    }
    __syncthreads();

    // ---- merge: the cell pairs of this block's cells ----
    // A cell belongs to a block by its representative: the blocks filled their
    // hashes each in its own order, so slots and list places mean nothing to
    // another block.
    uint16_t *own_cell = S.pos;
    for (int c = tid; c < ncells; c += NT) {
        const int r = S.rep[S.cell[c]];
        if (r != DB_NONE && (r & (NB - 1)) == rank) own_cell[atomicAdd(&S.nown, 1)] = S.cell[c];
    }
    __syncthreads();
    const int npairs = S.nown * noff;
    for (int k = tid; k < npairs; k += NT) {
        const int c = k / noff, sa = own_cell[c], ra = S.rep[sa];
        const unsigned keyA = S.key[sa];
        unsigned key;
        if (!key_at((int)(keyA % (unsigned)G), (int)((keyA / (unsigned)G) % (unsigned)G),
                    (int)(keyA / ((unsigned)G * (unsigned)G)), S.off[k - c * noff], G, key) ||
            key <= keyA)  // each cell pair from its smaller key
            continue;
        const int sb = find_cell(S, key, a.hbits);
        if (sb < 0 || S.rep[sb] == DB_NONE) continue;
        const unsigned rga = S.range[sa], rgb = S.range[sb];
        const int a0 = (int)(rga >> 16), a1 = a0 + (int)(rga & 0xffffu), b0 = (int)(rgb >> 16),
                  b1 = b0 + (int)(rgb & 0xffffu);
        bool hit = false, all = true;
        int tests = 0;
        for (int qa = a0; qa < a1 && !hit && all; ++qa) {
            if (!S.score[qa]) continue;
            const float4 pa = S.pt[qa];
            for (int qb = b0; qb < b1; ++qb) {
                if (!S.score[qb]) continue;
                if (++tests > kThreadTests) {
                    all = false;
                    break;
                }
                if (near(Tp1 + pa.w, 2.f * pa.x, 2.f * pa.y, 2.f * pa.z, S.pt[qb])) {
                    hit = true;
                    break;
                }
            }
        }
        if (!hit && !all) {  // many pairs: a warp takes it, or this thread when the list is full
            const int at2 = atomicAdd(&S.nlist, 1);
            if (at2 < kList) {
                S.list[at2] = ((unsigned)sa << 16) | (unsigned)sb;
            } else {
                for (int qa = a0; qa < a1 && !hit; ++qa) {
                    if (!S.score[qa]) continue;
                    const float4 pa = S.pt[qa];
                    for (int qb = b0; qb < b1 && !hit; ++qb)
                        if (S.score[qb]) {
                            ++tests;
                            hit = near(Tp1 + pa.w, 2.f * pa.x, 2.f * pa.y, 2.f * pa.z, S.pt[qb]);
                        }
                }
            }
        }
        ev_merge += (unsigned)tests;
        if (hit) db::uf_unite(a.parent, ra, S.rep[sb], a.status);
    }
    __syncthreads();
    for (int e = wid; e < min(S.nlist, kList); e += NT / 32) {
        const int sa = (int)(S.list[e] >> 16), sb = (int)(S.list[e] & 0xffffu);
        int same = 0;
        if (lane == 0) same = db::uf_find(a.parent, S.rep[sa]) == db::uf_find(a.parent, S.rep[sb]);
        if (__shfl_sync(FULL, same, 0)) continue;
        const unsigned rga = S.range[sa], rgb = S.range[sb];
        const int a0 = (int)(rga >> 16), a1 = a0 + (int)(rga & 0xffffu), b0 = (int)(rgb >> 16),
                  b1 = b0 + (int)(rgb & 0xffffu);
        bool hit = false;
        for (int x0 = a0; x0 < a1 && !hit; x0 += 32) {
            const int qa = x0 + lane;
            const bool on = qa < a1 && S.score[qa];
            const unsigned rows = __ballot_sync(FULL, on);
            if (!rows) continue;
            const float4 pa = S.pt[on ? qa : a0];
            for (int qb = b0; qb < b1 && !hit; ++qb) {
                if (!S.score[qb]) continue;
                if (lane == 0) ev_merge += (unsigned)__popc(rows);
                hit = __any_sync(FULL, on && near(Tp1 + pa.w, 2.f * pa.x, 2.f * pa.y, 2.f * pa.z, S.pt[qb]));
            }
        }
        if (hit && lane == 0) db::uf_unite(a.parent, S.rep[sa], S.rep[sb], a.status);
        __syncwarp();
    }

    // ---- border: the smallest-index core neighbour of this block's other points ----
    int best = DB_NONE, bslot = A;
    const bool core = mine && S.core[i];
    if (mine && !core) {
        best = S.rep[A];
        for (int o = 0; o < noff; ++o) {
            unsigned key;
            if (!key_at(cx, cy, cz, S.off[o], G, key)) continue;
            const int B = find_cell(S, key, a.hbits);
            if (B < 0 || S.rep[B] >= best) continue;  // no core index of B can beat the current best
            const unsigned r = S.range[B];
            const int q0 = (int)(r >> 16), q1 = q0 + (int)(r & 0xffffu);
            for (int q = q0; q < q1; ++q) {
                if (!S.score[q] || S.idx[q] >= best) continue;
                ++ev_border;
                if (near(cp, px2, py2, pz2, S.pt[q])) {
                    best = S.idx[q];
                    bslot = B;
                }
            }
        }
    }
    cluster_arrive();
    cluster_wait();  // the forest is complete

    // ---- labels ----
    int lab = -1, kind = -1;
    bool root = false;
    if (mine) {
        kind = core ? 0 : (best != DB_NONE ? 1 : 2);
        if (kind != 2) lab = db::uf_find(a.parent, S.rep[bslot]);
        root = core && lab == i;
    }
    if (a.compact) {  // rank of each root: every block marks all of them
        for (int w = tid; w <= kMaxN / 32; w += NT) S.bits[w] = 0u;
        __syncthreads();
        for (int c = tid; c < ncells; c += NT) {
            const int r = S.rep[S.cell[c]];
            if (r != DB_NONE && db::ld_relaxed(a.parent + r) == r) atomicOr(&S.bits[r >> 5], 1u << (r & 31));
        }
        __syncthreads();
        if (wid == 0) {
            int base = 0;
            for (int w0 = 0; w0 < kMaxN / 32; w0 += 32) {
                const int v = __popc(S.bits[w0 + lane]);
                int inc = v;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const int y = __shfl_up_sync(FULL, inc, o);
                    if (lane >= o) inc += y;
                }
                S.before[w0 + lane] = base + inc - v;
                base += __shfl_sync(FULL, inc, 31);
            }
        }
        __syncthreads();
        if (lab >= 0) lab = S.before[lab >> 5] + __popc(S.bits[lab >> 5] & ((1u << (lab & 31)) - 1u));
    }
    if (mine) {
        a.labels[i] = lab;
        if (a.counts_out) a.counts_out[i] = count;
        if (a.core_out) a.core_out[i] = core;
    }

    // ---- statistics ----
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const unsigned m = __ballot_sync(FULL, k < 3 ? kind == k : root);
        if (lane == 0 && m) atomicAdd(&S.red[k], __popc(m));
    }
    __syncthreads();
    if (tid < 4 && S.red[tid]) atomicAdd(a.ctr + 2 + tid, (unsigned long long)S.red[tid]);
    if (rank == 0 && tid == 0) a.ctr[0] = ((unsigned long long)ncells << 32) | (unsigned)n;
    db::block_sum_add(a.ctr + DB_CTR_EVAL, ev_count);
    __syncthreads();
    db::block_sum_add(a.ctr + DB_CTR_EVAL + 1, ev_merge);
    __syncthreads();
    db::block_sum_add(a.ctr + DB_CTR_EVAL + 2, ev_border);
    __syncthreads();
    if (a.stats) db::block_sum_add(a.ctr + 1, cand);
}

}  // namespace

// Clears the counters itself, and the status word when `reset` is set.
cudaError_t launch_grid_small(const DbWork &w, const GridGeom &g, const float *x, int64_t n, int32_t min_pts, bool exact,
                              bool compact, bool stats, bool reset, int32_t *labels, int32_t *counts_out,
                              uint8_t *core_out, cudaStream_t st) {
    SmallArgs a{};
    a.x = x;
    a.n = (int)n;
    a.hbits = g.hbits;  // at least 10, at least 2 n slots
    a.min_pts = min_pts;
    a.exact = exact ? 1 : 0;
    a.compact = compact ? 1 : 0;
    a.stats = stats ? 1 : 0;
    a.reset = reset ? 1 : 0;
    a.g = g;
    a.parent = w.parent;
    a.labels = labels;
    a.counts_out = counts_out;
    a.core_out = core_out;
    a.status = w.status;
    a.ctr = w.ctr;
    if ((1 << a.hbits) > kSlots || g.noff > 124) return cudaErrorInvalidValue;
    cudaError_t e = cudaFuncSetAttribute(grid_small_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)sizeof(SmallSmem));
    if (e) return e;
    grid_small_kernel<<<NB, NT, sizeof(SmallSmem), st>>>(a);
    w.marks->kernel("grid_small", st);
    return cudaGetLastError();
}
