// grid_small.cu — the eps-grid path for small point sets (d <= 3, up to 2,048
// points), in one launch.
//
// The grid path (grid.cu) is a chain of some ten kernels; with a few thousand
// points each of them works for a microsecond or two, and the launches, the
// clears and the gaps between them are what a call takes (2,000 points in the
// plane: 99 us a call, 70 with the merge on a forest in global memory, 60 on
// forests in shared memory, 50 with the status written to the host by the kernel).  Here one thread block cluster runs the whole method: every block
// bins all points into its own shared memory (the binning is cheaper than
// sharing it) and counts neighbours and finds border neighbours for its eighth
// of the points.  The blocks meet when the core flags are known (each block
// writes its points' flags into every block's shared memory), and again after
// the merge: each tests the cell pairs of its eighth of the cells on a forest of
// its own in shared memory, then takes over the other blocks' links, one parent
// a set and block.  One forest in global memory, with eight blocks linking the
// same few roots, took 25 us of the call; all pairs in every block took 58.
//
// The limit: on eight SMs the time grows with n, on the whole chip it hardly does.
// Calls on the field recipe, this kernel / the chain of grid_rows.cu: 1,000
// points 50 / 84 us in the plane and 66 / 92 in space, 2,000 71 / 91 and 94 / 101,
// 2,500 81 / 84 and 104 / 103, 4,096 108 / 90 and 130 / 106.
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

constexpr int kMaxN = kGridSmallMaxN;  // 2,048
constexpr int NB = 8, NT = 512;        // blocks of the cluster, threads of a block: at most one own point a thread
constexpr int kSlots = 2 * kMaxN;      // cell hash
constexpr int kList = 2048;            // merge: cell pairs in two sets, a warp each
constexpr int kHookSteps = 4;          // merge: steps of 32 tests for a cell and one neighbour when it is hooked
constexpr float kFar = -1e30f;         // near nothing
constexpr unsigned FULL = 0xffffffffu;
static_assert(kList * sizeof(unsigned) >= kMaxN * sizeof(uint16_t), "the list's place holds a forest");

struct SmallSmem {
    float4 pt[kMaxN];         // {u0, u1, u2, -|u|^2} grouped by cell; from the merge on w = kFar if not core
    unsigned key[kSlots];     // cell hash
    unsigned range[kSlots];   // (first position << 16) | points of the cell
    int rep[kSlots];          // smallest core index of the cell (first: fill cursor)
    unsigned list[kList];     // (slot << 16) | slot; then the forest after this block's pairs
    uint16_t cell[kMaxN];     // slots of the occupied cells
    uint16_t idx[kMaxN];      // point at each position
    uint16_t pos[kMaxN];      // position of each point; then this block's cells in the merge
    uint16_t slot[kMaxN];     // cell of each position
    uint16_t par[kMaxN];      // forest, by point
    uint8_t core[kMaxN];      // by point (written by all blocks)
    char4 off[128];
    int wsum[NT / 32], wocc[NT / 32];
    unsigned other[NT];       // this block's other points: (position << 16) | thread
    unsigned found[NT];       // (smallest core neighbour << 16) | its cell's slot, by thread
    unsigned bits[kMaxN / 32 + 1];  // roots: those that the hooking left, then those of the labels
    int before[kMaxN / 32 + 1];
    int nlist, nown, nother;
    int red[4];
};

struct SmallArgs {
    const float *x;
    int n, hbits, min_pts, exact, compact, stats, reset;
    GridGeom g;
    int *labels, *counts_out;
    uint8_t *core_out;
    unsigned *status, *status_out;
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

// Union-find over point indices in shared memory.
__device__ __forceinline__ int find_root(volatile uint16_t *par, int x) {
    while (true) {
        const int p = par[x];
        if (p == x) return x;
        const int gp = par[p];
        if (gp == p) return p;
        par[x] = (uint16_t)gp;
        x = gp;
    }
}
__device__ __forceinline__ void unite(uint16_t *par, int a, int b, unsigned *status) {
    for (int it = 0; it < (1 << 20); ++it) {
        a = find_root(par, a);
        b = find_root(par, b);
        if (a == b) return;
        if (a > b) {
            const int t = a;
            a = b;
            b = t;
        }
        if (atomicCAS(reinterpret_cast<unsigned short *>(par + b), (unsigned short)b, (unsigned short)a) == b) return;
    }
    atomicOr(status, DB_EBIT_TIMEOUT);
}

// The cells at four offsets, their first probes side by side (-1: none).
struct Four {
    int slot[4];
};
__device__ __forceinline__ Four find_four(const SmallSmem &S, int cx, int cy, int cz, int o, int noff, int G, int bits) {
    const unsigned mask = (1u << bits) - 1u;
    Four f;
    unsigned key[4], h[4], k[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        const char4 off = S.off[min(o + u, noff - 1)];
        const int x = cx + off.x, y = cy + off.y, z = cz + off.z;
        const bool in = o + u < noff && x >= 0 && x < G && y >= 0 && y < G && z >= 0 && z < G;
        key[u] = ((unsigned)z * (unsigned)G + (unsigned)y) * (unsigned)G + (unsigned)x;
        h[u] = db::hash_slot(key[u], bits) & mask;
        k[u] = in ? S.key[h[u]] : DB_HASH_EMPTY;
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        for (unsigned probe = 0; probe <= mask && k[u] != key[u] && k[u] != DB_HASH_EMPTY; ++probe) {
            h[u] = (h[u] + 1) & mask;
            k[u] = S.key[h[u]];
        }
        f.slot[u] = k[u] == key[u] && k[u] != DB_HASH_EMPTY ? (int)h[u] : -1;
    }
    return f;
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

// Is a core point of cell a near one of cell b?  By GL lanes (`mask`), each with a
// point of the larger cell, against four points of the smaller a step; at most
// max_steps steps, then false with `all` cleared.
template <int GL>
__device__ __forceinline__ bool cells_near(const SmallSmem &S, float Tp1, int sa, int sb, int sub, unsigned mask,
                                           int max_steps, bool &all, unsigned long long &tests) {
    unsigned ra = S.range[sa], rb = S.range[sb];
    if ((ra & 0xffffu) < (rb & 0xffffu)) {
        const unsigned t = ra;
        ra = rb;
        rb = t;
    }
    const int a0 = (int)(ra >> 16), a1 = a0 + (int)(ra & 0xffffu), b0 = (int)(rb >> 16), b1 = b0 + (int)(rb & 0xffffu);
    int steps = 0;
    for (int x0 = a0; x0 < a1; x0 += GL) {
        const float4 pa = S.pt[min(x0 + sub, a1 - 1)];  // past the end: the last point again
        const float cp = Tp1 + pa.w, px2 = 2.f * pa.x, py2 = 2.f * pa.y, pz2 = 2.f * pa.z;
        for (int y0 = b0; y0 < b1; y0 += 4) {
            if (steps++ == max_steps) {
                all = false;
                return false;
            }
            bool hit = false;
#pragma unroll
            for (int u = 0; u < 4; ++u) hit |= near(cp, px2, py2, pz2, S.pt[min(y0 + u, b1 - 1)]);
            if (x0 + sub < a1) tests += (unsigned)min(4, b1 - y0);
            if (__ballot_sync(mask, hit) & mask) return true;
        }
    }
    return false;
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
    if (tid == 0) S.nlist = S.nown = S.nother = 0;
    for (int q = tid; q < n; q += NT) S.par[q] = (uint16_t)q;
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

    // ---- neighbour counts of this block's points: a group of lanes each ----
    const int own = (n + NB - 1) / NB;
    int gl = 0;  // log2 of the group, as many lanes as there are threads for
    while (gl < 3 && (own << (gl + 1)) <= NT) ++gl;
    const int sub = tid & ((1 << gl) - 1), local = tid >> gl, i = rank * own + local;
    const bool has = local < own && i < n, mine = has && sub == 0;
    float4 p = make_float4(0.f, 0.f, 0.f, 0.f);
    int A = 0, at_i = 0, cx = 0, cy = 0, cz = 0, count = 0;
    unsigned long long ev_count = 0, ev_merge = 0, ev_border = 0, cand = 0;
    if (has) {
        at_i = S.pos[i];
        p = S.pt[at_i];
        A = S.slot[at_i];
        const unsigned keyA = S.key[A];
        cx = (int)(keyA % (unsigned)G);
        cy = (int)((keyA / (unsigned)G) % (unsigned)G);
        cz = (int)(keyA / ((unsigned)G * (unsigned)G));
        count = (int)(S.range[A] & 0xffffu);  // the cell is a clique
    }
    const int lim = a.exact ? INT_MAX : a.min_pts;
    {
        const float cp = Tp1 + p.w, px2 = 2.f * p.x, py2 = 2.f * p.y, pz2 = 2.f * p.z;
        if (mine) cand = (unsigned)count;
        for (int o0 = 0; o0 < noff; o0 += 4 << gl) {
            // a group goes on while its point needs it: every lane has the group's count
            const bool go = has && (count < lim || a.stats);
            if (!__any_sync(FULL, go)) break;
            int add = 0;
            const int o = o0 + 4 * sub;
            if (go && o < noff) {
                const Four f = find_four(S, cx, cy, cz, o, noff, G, a.hbits);
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    if (f.slot[u] < 0) continue;
                    const unsigned r = S.range[f.slot[u]];
                    const int q0 = (int)(r >> 16), q1 = q0 + (int)(r & 0xffffu);
                    cand += r & 0xffffu;
                    if (count + add >= lim) continue;
                    int q = q0;
                    while (q < q1 && count + add < lim) {  // (a tight blob's cell: not all of it)
                        const int qe = min(q + 32, q1);
#pragma unroll 4
                        for (; q < qe; ++q) add += near(cp, px2, py2, pz2, S.pt[q]);
                    }
                    ev_count += (unsigned)(q - q0);
                }
            }
            __syncwarp();
            for (int b = 1; b < 1 << gl; b <<= 1) add += __shfl_xor_sync(FULL, add, b);
            count += add;
        }
    }
    cluster_wait();
    if (mine)
        for (int r = 0; r < NB; ++r) cluster.map_shared_rank(S.core, r)[i] = count >= a.min_pts;
    cluster_arrive();
    cluster_wait();  // core flags and the cleared counters are everywhere
    if (!ok) atomicOr(a.status, DB_EBIT_NOT_QUANTISED);

    // ---- representatives, by every block ----
    for (int q = tid; q < n; q += NT) {
        const int o = S.idx[q];
        const uint8_t c = S.core[o];
        if (c)
            atomicMin(&S.rep[S.slot[q]], o);
        else
            S.pt[q].w = kFar;
    }
    __syncthreads();

    // ---- merge ----
    // This block's cells (dealt out by their smallest core index: the hash of
    // each block fills in its own order) and its points that are not core.
    uint16_t *own_cell = S.pos, *par = S.par;
    for (int c = tid; c < ncells; c += NT) {
        const int r = S.rep[S.cell[c]];
        if (r != DB_NONE && (r & (NB - 1)) == rank) own_cell[atomicAdd(&S.nown, 1)] = S.cell[c];
    }
    for (int w = tid; w <= kMaxN / 32; w += NT) S.bits[w] = 0u;
    const bool core = mine && S.core[i];
    if (mine && !core) S.other[atomicAdd(&S.nother, 1)] = ((unsigned)at_i << 16) | (unsigned)tid;
    __syncthreads();
    // First every cell is hooked to one adjacent cell of smaller key, in all
    // blocks' forests at once: no exchange, and dense sets come down to a few
    // roots, where linking pair by pair has all threads at the same few.
    {
        const int sub8 = lane & 7;
        const unsigned mask = 0xffu << (lane & 24);
        for (int c = tid >> 3; c < S.nown; c += NT / 8) {
            const int sa = own_cell[c];
            const unsigned keyA = S.key[sa];
            const int ax = (int)(keyA % (unsigned)G), ay = (int)((keyA / (unsigned)G) % (unsigned)G),
                      az = (int)(keyA / ((unsigned)G * (unsigned)G));
            bool hit = false;
            for (int o0 = 0; o0 < a.g.nnear && !hit; o0 += 8) {  // a lane looks one neighbour up
                unsigned key;
                int mb = -1;
                if (o0 + sub8 < a.g.nnear && key_at(ax, ay, az, S.off[o0 + sub8], G, key) && key < keyA)
                    mb = find_cell(S, key, a.hbits);
                if (mb >= 0 && S.rep[mb] == DB_NONE) mb = -1;
                for (unsigned left = __ballot_sync(mask, mb >= 0) & mask; left && !hit; left &= left - 1) {
                    const int sb = __shfl_sync(mask, mb, __ffs(left) - 1);
                    bool all = true;
                    hit = cells_near<8>(S, Tp1, sa, sb, sub8, mask, kHookSteps, all, ev_merge);
                    if (hit) cluster.map_shared_rank(par, sub8)[S.rep[sa]] = (uint16_t)S.rep[sb];
                }
            }
        }
        __syncwarp();
    }
    cluster_arrive();
    cluster_wait();
    for (int c = tid; c < ncells; c += NT) {
        const int r = S.rep[S.cell[c]];
        if (r != DB_NONE) {
            const int root = find_root(par, r);
            if (root != r)
                *(volatile uint16_t *)(par + r) = (uint16_t)root;
            else
                atomicOr(&S.bits[r >> 5], 1u << (r & 31));
        }
    }
    __syncthreads();
    // Then the cell pairs of this block's cells that are in two sets yet, on its
    // own forest, the adjacent ones first.
    for (int ring = 0; ring < 2; ++ring) {
        const int o0 = ring ? a.g.nnear : 0, no = (ring ? noff : a.g.nnear) - o0, npairs = S.nown * no;
        for (int k0 = 0; k0 < npairs; k0 += kList) {
            __syncthreads();
            if (tid == 0) S.nlist = 0;
            __syncthreads();
            for (int k = k0 + tid; k < min(k0 + kList, npairs); k += NT) {
                const int c = k / no, sa = own_cell[c];
                const unsigned keyA = S.key[sa];
                unsigned key;
                if (!key_at((int)(keyA % (unsigned)G), (int)((keyA / (unsigned)G) % (unsigned)G),
                            (int)(keyA / ((unsigned)G * (unsigned)G)), S.off[o0 + k - c * no], G, key) ||
                    key <= keyA)  // each cell pair from its smaller key
                    continue;
                const int sb = find_cell(S, key, a.hbits);
                if (sb < 0 || S.rep[sb] == DB_NONE || find_root(par, S.rep[sa]) == find_root(par, S.rep[sb])) continue;
                S.list[atomicAdd(&S.nlist, 1)] = ((unsigned)sa << 16) | (unsigned)sb;
            }
            __syncthreads();
            for (int e = wid; e < S.nlist; e += NT / 32) {
                const int sa = (int)(S.list[e] >> 16), sb = (int)(S.list[e] & 0xffffu);
                const int same = lane == 0 && find_root(par, S.rep[sa]) == find_root(par, S.rep[sb]);
                if (__shfl_sync(FULL, same, 0)) continue;
                bool all = true;
                if (cells_near<32>(S, Tp1, sa, sb, lane, FULL, INT_MAX, all, ev_merge) && lane == 0)
                    unite(par, S.rep[sa], S.rep[sb], a.status);
                __syncwarp();
            }
        }
    }

    // The other blocks read a copy: this block goes on linking, and a parent
    // that is shortened past a link they have not seen would lose the set between.
    __syncthreads();
    uint16_t *links = reinterpret_cast<uint16_t *>(S.list);
    for (int q = tid; q < n; q += NT) links[q] = par[q];
    cluster_arrive();

    // ---- border: the smallest-index core neighbour of this block's other
    // points, a warp each and a lane a neighbour cell ----
    for (int e = wid; e < S.nother; e += NT / 32) {
        const unsigned ent = S.other[e];
        const float4 pe = S.pt[ent >> 16];  // not core: its w is gone
        const float cp = Tp1 - (pe.x * pe.x + pe.y * pe.y + pe.z * pe.z);
        const int sa = S.slot[ent >> 16];
        const unsigned keyA = S.key[sa];
        const int ax = (int)(keyA % (unsigned)G), ay = (int)((keyA / (unsigned)G) % (unsigned)G),
                  az = (int)(keyA / ((unsigned)G * (unsigned)G));
        int best = S.rep[sa], bslot = sa;
        for (int o = lane; o < noff; o += 32) {
            unsigned key;
            if (!key_at(ax, ay, az, S.off[o], G, key)) continue;
            const int B = find_cell(S, key, a.hbits);
            if (B < 0 || S.rep[B] >= best) continue;  // no core index of B can beat the current best
            const unsigned r = S.range[B];
            const int q0 = (int)(r >> 16), q1 = q0 + (int)(r & 0xffffu);
            for (int q = q0; q < q1; ++q) {
                if (S.idx[q] >= best) continue;
                ++ev_border;
                if (near(cp, 2.f * pe.x, 2.f * pe.y, 2.f * pe.z, S.pt[q])) {
                    best = S.idx[q];
                    bslot = B;
                }
            }
        }
        __syncwarp();
        const unsigned low = __reduce_min_sync(
            FULL, best == DB_NONE ? 0xffffffffu : ((unsigned)best << 16) | (unsigned)bslot);
        if (lane == 0) S.found[ent & 0xffffu] = low;
    }

    // ---- the other blocks' links, where they can differ: at the roots that the
    // hooking left (with all cells' parents, hundreds of threads tried the same
    // few links, 25,000 cycles) ----
    cluster_wait();
    for (int c = tid; c < ncells; c += NT) {
        const int r = S.rep[S.cell[c]];
        if (r == DB_NONE || !(S.bits[r >> 5] >> (r & 31) & 1u)) continue;
        int up[NB];
#pragma unroll
        for (int o = 1; o < NB; ++o)
            up[o] = cluster.map_shared_rank(links, (rank + o) & (NB - 1))[r];
#pragma unroll
        for (int o = 1; o < NB; ++o)
            if (up[o] != r) unite(par, r, up[o], a.status);
    }
    cluster_arrive();  // waited for at the end: no block leaves while its links are read

    // ---- labels: the smallest core index of each set ----
    int *least = reinterpret_cast<int *>(S.range);  // by root (the cells are not looked at any more)
    for (int q = tid; q < n; q += NT) least[q] = DB_NONE;
    for (int w = tid; w <= kMaxN / 32; w += NT) S.bits[w] = 0u;
    __syncthreads();
    for (int c0 = 0; c0 < ncells; c0 += NT) {
        const int c = c0 + tid, r = c < ncells ? S.rep[S.cell[c]] : DB_NONE;
        const int root = r != DB_NONE ? find_root(par, r) : -1;
        const unsigned on = __ballot_sync(FULL, root >= 0);
        if (!on) continue;
        const int root0 = __shfl_sync(FULL, root, __ffs(on) - 1);  // most warps see one set
        const unsigned same = __ballot_sync(FULL, root == root0);
        const int low = (int)__reduce_min_sync(FULL, root == root0 ? (unsigned)r : 0xffffffffu);
        if (root == root0 ? lane == __ffs(same) - 1 : root >= 0) atomicMin(&least[root], root == root0 ? low : r);
    }
    __syncthreads();
    int lab = -1, kind = -1;
    bool root = false;
    if (mine) {
        const unsigned f = core ? 0u : S.found[tid];
        kind = core ? 0 : (f != 0xffffffffu ? 1 : 2);
        if (kind != 2) lab = least[find_root(par, S.rep[core ? A : (int)(f & 0xffffu)])];
        root = core && lab == i;
    }
    if (a.compact) {  // rank of each root: every block marks all of them
        for (int c = tid; c < ncells; c += NT) {
            const int r = S.rep[S.cell[c]];
            if (r != DB_NONE && least[find_root(par, r)] == r) atomicOr(&S.bits[r >> 5], 1u << (r & 31));
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
    cluster_wait();
    db::report_status(a.status, a.status_out);  // no block sets a bit after its arrival
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
    a.labels = labels;
    a.counts_out = counts_out;
    a.core_out = core_out;
    a.status = w.status;
    a.status_out = w.status_out;
    a.ctr = w.ctr;
    if ((1 << a.hbits) > kSlots || g.noff > 124) return cudaErrorInvalidValue;
    cudaError_t e = cudaFuncSetAttribute(grid_small_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)sizeof(SmallSmem));
    if (e) return e;
    grid_small_kernel<<<NB, NT, sizeof(SmallSmem), st>>>(a);
    w.marks->kernel("grid_small", st);
    return cudaGetLastError();
}
