// internal.cuh — shared device helpers and launch declarations of libdbscan_gb300.
//
// Notation follows the paper (Wang et al., Sections II and IV): a point p has
// grid units u_p (integers 0..1023), T = floor(eps^2 * 2^20) and q is an
// eps-neighbour of p iff D(p,q) = sum_k (u_pk - u_qk)^2 <= T.
#pragma once

#include <utility>

#include <cuda_runtime.h>
#include <stdint.h>

#include "dbscan.h"  // include/ is on the include path

// Device-side error bits, OR-ed into the plan's status word.
#define DB_EBIT_NOT_QUANTISED 1u
#define DB_EBIT_TIMEOUT 2u     // a bounded loop gave up
#define DB_EBIT_OVERFLOW 4u    // a device-side list ran out of room

#define DB_NONE 0x7fffffff     // "no index" (larger than every point index)

// Device counters of a run (DbWork::ctr, DB_NCTR 64-bit slots):
//   0 grid cells|points, 1 grid candidate pairs, 2..5 core/border/noise/clusters,
//   6 band pairs rechecked, 7..8 band verification, 9..13 and 20..29 pipeline
//   diagnostics of the tensor-core count, merge and border passes,
//   15 FP16 tensor-core count ran the folded form (1),
//   16..19 pair tests evaluated by the count, merge, border and (grid path)
//   outer-ring merge passes, 30 cell pairs left to the eps-grid's search (int),
//   31 work items of the projected grid (int).
#define DB_NCTR 32
#define DB_CTR_EVAL 16
#define DB_CTR_TC_FOLD 15      // 1: the FP16 count ran the folded form
#define DB_CTR_PAIRS 30
#define DB_CTR_MID_ITEMS 31
#define DB_HASH_EMPTY 0xffffffffu

namespace db {

// ---------------------------------------------------------------------------
// Relaxed, L1-bypassing accesses for data other threads update concurrently.
// ---------------------------------------------------------------------------
__device__ __forceinline__ int ld_relaxed(const int *p) {
    int v;
    asm volatile("ld.relaxed.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void st_relaxed(int *p, int v) {
    asm volatile("st.relaxed.gpu.global.s32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

}  // namespace db

#include "union_find.cuh"

namespace db {

// Cell hash slot of the grid paths: four consecutive keys (four cells in a
// row along x) share one 32-byte bucket of the packed table, so the lookups of
// a cell's x-neighbours, made by neighbouring lanes, touch few sectors.
__device__ __forceinline__ unsigned hash_slot(unsigned key, int bits) {
    return ((((key >> 2) * 2654435761u) >> (34 - bits)) << 2) | (key & 3u);
}

// 2^-10 grid check of one coordinate: finite, 0 <= x < 1, 1024 x integral.
__device__ __forceinline__ bool on_grid(float x, int &u) {
    float s = x * 1024.0f;  // exact: scaling by a power of two
    bool ok = (x >= 0.0f) && (x < 1.0f) && (s == floorf(s));
    u = ok ? (int)s : 0;
    return ok;
}

// Sum of v over the block added to *dst by one global atomic.  Every thread
// of the block must call it (it synchronises the block).
__device__ __forceinline__ void block_sum_add(unsigned long long *dst, unsigned long long v) {
    __shared__ unsigned long long part[32];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x == 0) {
        unsigned long long t = 0;
        for (int w = 0; w < (int)((blockDim.x + 31) >> 5); ++w) t += part[w];
        if (t) atomicAdd(dst, t);
    }
}

// Programmatic dependent launch.  A kernel started with launch_dependent()
// may be scheduled while the kernel before it in its stream still runs: it
// calls wait_prior_grid() before touching memory, which returns once that
// kernel has completed and its writes are visible (at once for a kernel
// started the plain way).  allow_next_grid() lets the next such kernel of the
// stream be scheduled early; it still waits for this one to complete.  A
// chain of short dependent kernels then overlaps each launch with the tail of
// the kernel before it.
__device__ __forceinline__ void wait_prior_grid() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void allow_next_grid() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// The run's status word to the host, by the run's label kernel: every kernel that
// can set a bit has completed by then.  (With a copy behind the
// run instead, 2,000 points in the plane took 57.6 us a call, now 50.2; 6,007 x 32
// 134, now 128.)
__device__ __forceinline__ void report_status(const unsigned *status, unsigned *out) {
    if (out && blockIdx.x == 0 && threadIdx.x == 0)
        *(volatile unsigned *)out = (unsigned)ld_relaxed(reinterpret_cast<const int *>(status));
}

__device__ __forceinline__ unsigned lanemask_lt() {
    unsigned m;
    asm("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
    return m;
}

}  // namespace db

// Starts kern on st as a programmatic dependent of the previous kernel in st
// (kern must call db::wait_prior_grid() before its first memory access).
template <typename... P, typename... A>
inline cudaError_t launch_dependent_smem(void (*kern)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st,
                                         A &&...args) {
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, std::forward<A>(args)...);
}
template <typename... P, typename... A>
inline cudaError_t launch_dependent(void (*kern)(P...), dim3 grid, dim3 block, cudaStream_t st, A &&...args) {
    return launch_dependent_smem(kern, grid, block, 0, st, std::forward<A>(args)...);
}

// ---------------------------------------------------------------------------
// Per-kernel timing: when on, a CUDA event is recorded on the launch stream
// after every kernel, so kernel i took elapsed(ev[i-1] or start, ev[i]).
// ---------------------------------------------------------------------------
struct PhaseMarks {
    static constexpr int kMax = 32;
    bool on = false;
    int n = 0;
    int kernels = 0;
    cudaEvent_t start = nullptr;
    cudaEvent_t ev[kMax] = {};
    const char *name[kMax] = {};
    void begin(cudaStream_t st) {
        n = 0;
        kernels = 0;
        if (on) cudaEventRecord(start, st);
    }
    void kernel(const char *nm, cudaStream_t st) {
        ++kernels;
        if (on && n < kMax) {
            cudaEventRecord(ev[n], st);
            name[n++] = nm;
        }
    }
};

// ---------------------------------------------------------------------------
// Workspace of one clustering run (device pointers carved from one allocation).
// ---------------------------------------------------------------------------
struct DbWork {
    int64_t cap_n;
    int32_t cap_d;
    int32_t dp_cap;         // padded row stride capacity of P
    // all paths
    float *P;               // packed grid units, row stride DP (all-pairs) [cap_n * dp_cap]
    int32_t *count;         // neighbour counts by point index [cap_n]
    uint8_t *core;          // core flags by point index [cap_n]
    int32_t *parent;        // union-find forest by point index [cap_n]
    int32_t *border;        // smallest core neighbour of non-core points [cap_n]
    int32_t *scan;          // exclusive-scan output [cap_n + 1]
    int32_t *scan_part;     // scan partials
    int64_t scan_part_cap;
    unsigned *status;       // device error bits
    unsigned long long *ctr;  // DB_NCTR counters (slots listed beside DB_NCTR)
    unsigned *status_out;     // pinned host word for a run that is waited for (null: none), see report_status
    // grid path
    int64_t hcap;           // hash slots (power of two >= 2 cap_n)
    int32_t hbits;
    uint32_t *hkey;
    int32_t *hcount;
    int2 *hpack;            // cell hash: {key, cell id} (written after the inserts) [hcap]
    uint32_t *occ;          // occupancy bitmap of all G^d cells, when it fits [occ_cap]
    int64_t occ_cap;        // words (128 bits per point, at least 2^20 bits)
    int32_t *hcursor;
    int32_t *slot_of;       // hash slot of each point [cap_n]
    float4 *pts4;           // {u0,u1,u2,-|u|^2} by point index [cap_n]
    float4 *spts;           // same, grouped by cell [cap_n]
    int32_t *sidx;          // point index of each grouped position [cap_n]
    int32_t *scell;         // cell id of each grouped position [cap_n]
    uint8_t *score;         // core flag of each grouped position [cap_n]
    int32_t *cell_start, *cell_count, *cell_rep;  // [cap_n]
    float4 *cell_mid;       // a core point near each cell's centre [cap_n]
    uint32_t *cell_key;     // [cap_n]
    int32_t *nbr;           // neighbour cell lists, adjacent first [cap_n * noff_cap]
    int32_t *ncnt;          // (adjacent count << 16) | count [cap_n]
    int32_t *cell_cand;     // points in the cells of each neighbour list [cap_n]
    int32_t noff_cap;
    uint2 *rk;              // cells in key order: per 32 cells {occupied cells before, bits} [occ_cap] (over hpack and on)
    unsigned long long *rg_part;  // block totals of its scans
    // tensor-core path (max_d >= 16)
    int64_t tc_cap_pad;     // rows of each packed operand (cap_n rounded up to 256, plus 256)
    int16_t *v16;           // centred units by position, row stride K (BF16 recheck, verification) [cap_n * 64]
    uint16_t *opAll;        // packed operand tiles: FP16 with the folded chunk, or two BF16 terms [tc_cap_pad * 128]
    uint16_t *opCore, *opNon;  // FP16 tiles of the points before ordering; pivots, then ball centres [tc_cap_pad * 64]
    void *metaAll, *metaCore, *metaNon;  // per-tile metadata: all, core points only, border rows only (16 B per point)
    int32_t *list_a, *list_b;  // point of each position [tc_cap_pad], position of each point [cap_n]
    int32_t *tc_lens;       // [0] largest |v|^2
    int32_t *tc_hist;       // buckets of the order [8192]
    int32_t *tc_tag, *tc_rowneed, *tc_udone;  // per tile: common root of its core points, border rows; per unit
    float *tc_cbeta, *tc_crad;  // per ball (two a tile): |c|^2 of its centre, largest squared distance to it
    uint32_t *tc_pairs;     // tile pairs that may hold neighbours (bits) [tiles][ceil(tiles / 32)]
    void *wt;               // warp-tile path (d <= 16 all pairs): its arrays, over other paths' (null: not served)
    PhaseMarks *marks;      // host-side timing marks of the owning plan
    // second stream of the grid path: independent kernels run beside each
    // other (fork/join by events); unused while per-kernel marks are taken
    cudaStream_t side;
    cudaEvent_t fj[4];
};

// Host-side grid geometry for d <= 3 (see grid.cu).
struct GridGeom {
    int32_t d, c, G, Tc, noff, nnear, hbits;
    int32_t dense;  // 1: cells indexed directly by key (slot = key, G^d slots), 0: hashed (2^hbits slots)
    float Tp1;
    float inv_c;    // 1/c rounded to FP32: floor((u + 1/2) * inv_c) = floor(u / c) for 0 <= u < 2^11
    char4 off[124];
};

// ---- launchers (all enqueue on `st`; return cudaError_t of the launch) ----
cudaError_t launch_prep_dense(const DbWork &w, const float *x, int64_t n, int32_t d, int32_t dp, cudaStream_t st);
cudaError_t launch_allpairs_simt(const DbWork &w, int64_t n, int32_t d, int32_t dp, int64_t Tc, int32_t min_pts,
                                 bool exact_counts, cudaStream_t st);
cudaError_t launch_allpairs_tc(const DbWork &w, const float *x, int64_t n, int32_t d, int64_t Tc, int32_t min_pts,
                               bool exact, bool bf16, bool stall, int32_t *labels, int32_t *counts_out,
                               uint8_t *core_out, cudaStream_t st);
cudaError_t launch_tc_verify(const DbWork &w, const float *x, int64_t n, int32_t d, int64_t Tc, bool bf16,
                             cudaStream_t st);
// In-place exclusive scan of n bucket sizes by one block.
cudaError_t launch_bucket_scan(int32_t *v, int32_t n, cudaStream_t st);
// All pairs for d <= 16 on ordered rows (pairs_wt.cu): device bytes of its
// arrays, and the whole run.
constexpr int kWtMaxCellBits = 18;  // cells of its counting sort
size_t wt_bytes(int64_t n);
cudaError_t launch_allpairs_wt(const DbWork &w, const float *x, int64_t n, int32_t d, int64_t Tc, int32_t min_pts,
                               bool exact, int32_t *labels, int32_t *counts_out, uint8_t *core_out, cudaStream_t st);
cudaError_t launch_labels_allpairs(const DbWork &w, int64_t n, int32_t *labels, int32_t *counts_out,
                                   uint8_t *core_out, cudaStream_t st);
cudaError_t launch_compact(const DbWork &w, int64_t n, int32_t *labels, cudaStream_t st);
cudaError_t launch_exclusive_scan(const int32_t *in, int32_t *out, int64_t n, int32_t *part, int64_t part_cap,
                                  cudaStream_t st, PhaseMarks *pm);
bool grid_geometry(int32_t d, int64_t Tc, int64_t n, GridGeom *g);
cudaError_t launch_grid_path(const DbWork &w, const GridGeom &g, const float *x, int64_t n, int32_t min_pts,
                             bool exact_counts, int32_t *labels, int32_t *counts_out, uint8_t *core_out,
                             cudaStream_t st);
// The whole eps-grid run of up to kGridSmallMaxN points in one launch
// (grid_small.cu), labels dense when `compact`; clears the run's counters, and
// the status word when `reset` is set.
constexpr int kGridSmallMaxN = 2048;
cudaError_t launch_grid_small(const DbWork &w, const GridGeom &g, const float *x, int64_t n, int32_t min_pts, bool exact,
                              bool compact, bool stats, bool reset, int32_t *labels, int32_t *counts_out,
                              uint8_t *core_out, cudaStream_t st);
// The eps-grid run with cells in key order (grid_rows.cu): whether it serves an
// instance, and the run; clears the run's counters, and the status word when
// `reset` is set.
bool grid_rows_serves(const DbWork &w, const GridGeom &g, int64_t n);
cudaError_t launch_grid_rows(const DbWork &w, const GridGeom &g, const float *x, int64_t n, int32_t min_pts, bool exact,
                             bool stats, bool reset, int32_t *labels, int32_t *counts_out, uint8_t *core_out,
                             cudaStream_t st);
// Ordered candidate pairs of a grid run (own cell listed: the projected grid).
cudaError_t launch_grid_candidates(const DbWork &w, const GridGeom &g, int64_t n, bool own_cell_listed,
                                   cudaStream_t st);
// Structure kernels shared by the eps-grid and the projected grid (grid_mid.cu):
// occupied slots -> cell table (ids, ranges, keys, occupancy bits), and the
// neighbour-cell lists of g's offsets.
cudaError_t launch_grid_cells(const DbWork &w, const GridGeom &g, unsigned *occ, unsigned long long *midkey,
                              cudaStream_t st);
cudaError_t launch_grid_nbrs(const DbWork &w, const GridGeom &g, const unsigned *occ, cudaStream_t st);
// Projected grid for 4 <= d <= 8 (grid_mid.cu): geometry (false when the
// cells would be too coarse to prune) and the whole path.
bool mid_geometry(int32_t d, int64_t Tc, int64_t n, GridGeom *g);
cudaError_t launch_mid_grid_path(const DbWork &w, const GridGeom &g, const float *x, int64_t n, int32_t d,
                                 int32_t min_pts, bool exact_counts, int32_t *labels, int32_t *counts_out,
                                 uint8_t *core_out, cudaStream_t st);
cudaError_t launch_stats(const DbWork &w, int64_t n, const int32_t *labels, cudaStream_t st);
int32_t dp_for(int32_t d);
