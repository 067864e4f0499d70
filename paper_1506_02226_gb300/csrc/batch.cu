// batch.cu — many independent instances in one graph-captured launch sequence.
//
// Each instance is one DBSCAN problem (Section II's definitions, the three
// steps of Section IV) with its own n, d, eps and min_pts.  The instances are
// concatenated in tiles of 64 rows (an instance's last tile is padded).
// Instances of up to kSortMax points are put in Z-order, so that a tile covers
// a small region; every pass is one persistent kernel whose warps pull work
// items (half a tile, a chunk of column tiles) from an atomic counter and run
// the ordered pair test (warp_tile.cuh).  The kernel
// sequence (prep, count, core flags with the merge inside tiles, the merge
// across near tiles, roots, the rest of the merge, border, labels, optional
// compaction) is captured once into a CUDA graph; a batch is then one table
// upload and one graph launch.
//
// Measured, 4,096 instances of 64 to 8,192 points, d in {2, 3, 16} (us, kernels
// one by one; with 64 x 64 FP32 tiles a block, before / after): prep 1,874 / 604
// (scattered row reads, the counting sort), count 10,030 / 912, core flags and
// the merge inside tiles - / 349, the merge across tiles 30,161 / 1,344 (pairs of
// tiles that hold several sets or none of whose pairs are neighbours), border
// 4,556 / 852; 46.6 / 4.1 ms a batch.  All passes are bound by the latency of an item's
// first loads (record, rows, boxes) and then by the scores' FP32 operations, two
// a pair; the matrix instructions are a few percent of the issue slots.
// On a plan of DBSCAN_PREC_EXACT_SIMT the passes take their dot products on the
// CUDA cores: 16.1 ms for the same batch (46.6 as 64 x 64 FP32 tiles).
//
// Autotuning: the column chunk per work item (CH) and the number of resident
// blocks per SM are picked on the first call by timing every candidate on the
// caller's batch; the pick is kept by the plan.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>

#include "batch_items.h"
#include "plan.h"
#include "warp_tile.cuh"

using namespace wtile;

namespace {

static_assert(BT == batchitems::kTileRows, "rows of a tile");

struct BHdr {  // the sizes of a run, and the tiles before each step of its passes
    Hdr h;
    unsigned first[batchitems::kMaxSteps + 1];
};

struct BInst {
    const float *x;
    int32_t *labels;
    TileRec rec;
};

// One block per instance at a time.  An instance of 2 .. sort_cap points is
// put in Z-order of its first three grid coordinates, so that a 64-row tile
// covers a small region; larger ones keep their order.  The order is a counting
// sort over 2 n to 4 n cells of the Z curve (points of one cell in any order)
// with 16-bit counters in shared memory: two passes over the points and one
// over the counters (4,096 instances of 64 to 8,192 points: 0.64 ms; with a
// bitonic sort of {code, index} keys 1.35).  Then the rows are packed in that
// order with their norms, perm gets the point of each row, and each tile its
// box: the least and greatest unit of its rows on every axis.  The reordering
// changes no result: every pass decides the same pairs, and labels are by point
// index.
__global__ void __launch_bounds__(512) batch_sortpack_kernel(const BInst *__restrict__ t,
                                                             const Hdr *__restrict__ hdr, int sort_cap, PackOut w,
                                                             unsigned *status) {
    extern __shared__ unsigned cells[];  // 2 counters a word: 2 sort_cap words, then sort_cap 16-bit indices
    __shared__ int wsum[16];
    uint16_t *order = reinterpret_cast<uint16_t *>(cells + 2 * sort_cap);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nwarps = blockDim.x >> 5;
    const int count = hdr->count;
    bool bad = false;
    for (int i = blockIdx.x; i < count; i += gridDim.x) {
        const BInst I = t[i];
        const int n = I.rec.n, d = I.rec.d;
        const bool sorted = n > 1 && n <= sort_cap;
        if (sorted) {
            const int dz = d < 3 ? d : 3;
            int lg = 1;
            while ((1 << lg) < n) ++lg;  // n <= 2^lg
            // the most bits per axis that keep 2^(dz bits) cells within 2^(lg + 2)
            const int bits = min(10, (lg + 2) / dz), words = (1 << (dz * bits)) / 2;  // 2 counters a word
            for (int c = tid; c < max(words, 1); c += blockDim.x) cells[c] = 0u;
            __syncthreads();
#pragma unroll 4
            for (int s = tid; s < n; s += blockDim.x) {
                const unsigned c = zcode(I.x + (size_t)s * d, dz, bits);
                atomicAdd(&cells[c >> 1], 1u << (16 * (c & 1u)));
            }
            __syncthreads();
            // exclusive starts: each thread a run of words, then the block
            const int per = (max(words, 1) + (int)blockDim.x - 1) / (int)blockDim.x;
            const int w0 = min(tid * per, max(words, 1)), w1 = min(w0 + per, max(words, 1));
            int sum = 0;
            for (int c = w0; c < w1; ++c) sum += (int)(cells[c] & 0xffffu) + (int)(cells[c] >> 16);
            int incl = sum;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += y;
            }
            if (lane == 31) wsum[warp] = incl;
            __syncthreads();
            int at = incl - sum;
            for (int k = 0; k < warp; ++k) at += wsum[k];
            for (int c = w0; c < w1; ++c) {
                const unsigned two = cells[c];
                cells[c] = (unsigned)at | ((unsigned)(at + (int)(two & 0xffffu)) << 16);
                at += (int)(two & 0xffffu) + (int)(two >> 16);
            }
            __syncthreads();
#pragma unroll 4
            for (int s = tid; s < n; s += blockDim.x) {
                const unsigned c = zcode(I.x + (size_t)s * d, dz, bits);
                const unsigned old = atomicAdd(&cells[c >> 1], 1u << (16 * (c & 1u)));
                order[(old >> (16 * (c & 1u))) & 0xffffu] = (uint16_t)s;
            }
            __syncthreads();
        }
        for (int tt = warp; tt < I.rec.ntiles; tt += nwarps)
            bad |= pack_tile_d(I.x, I.rec, tt, sorted ? order : nullptr, w);
        __syncthreads();  // the order is free again
    }
    if (bad) atomicOr(status, DB_EBIT_NOT_QUANTISED);
}

// Labels in each instance's own index space, a thread per row: a core row the
// smallest point index of its set, a border row that of its smallest-index
// core neighbour, noise -1; per-instance counts (core, border, noise,
// clusters) when istats != nullptr; root flags for compaction, by point.
__global__ void __launch_bounds__(NT) batch_label_kernel(Rows R, const Hdr *__restrict__ hdr,
                                                         const BInst *__restrict__ t, const int *__restrict__ inv,
                                                         const int *__restrict__ least, int *__restrict__ flags,
                                                         int *istats) {
    const int total = hdr->total_tiles * BT;
    for (int g = (int)(blockIdx.x * blockDim.x + threadIdx.x); g < total; g += (int)(gridDim.x * blockDim.x)) {
        const TileRec &I = R.tiles[g >> 6];
        if (g - I.tile0 * BT >= I.n) continue;
        const int loc = R.perm[g], bo = R.border[g];
        int lab = -1, kind = 2;
        if (R.core[g]) {
            lab = least[R.parent[g]];
            kind = 0;
        } else if (bo != DB_NONE) {
            lab = least[R.parent[inv[I.point0 + bo]]];
            kind = 1;
        }
        t[I.inst].labels[loc] = lab;
        const int root = (kind == 0 && lab == loc);
        if (flags) flags[I.point0 + loc] = root;
        if (istats) {
            atomicAdd(istats + 4 * I.inst + kind, 1);
            if (root) atomicAdd(istats + 4 * I.inst + 3, 1);
        }
    }
}

// Dense cluster numbers from the scan of the root flags (a thread per row).
__global__ void batch_compact_kernel(Rows R, const Hdr *__restrict__ hdr, const BInst *__restrict__ t,
                                     const int *__restrict__ rank) {
    const int total = hdr->total_tiles * BT;
    for (int g = (int)(blockIdx.x * blockDim.x + threadIdx.x); g < total; g += (int)(gridDim.x * blockDim.x)) {
        const TileRec &I = R.tiles[g >> 6];
        if (g - I.tile0 * BT >= I.n) continue;
        int *labels = t[I.inst].labels + R.perm[g];
        const int l = *labels;
        if (l >= 0) *labels = rank[I.point0 + l] - rank[I.point0];
    }
}

constexpr int kCH[] = {64, 256};
constexpr int kBPS[] = {4, 8};
static_assert(kCH[0] == batchitems::kMinChunk && kCH[1] % kCH[0] == 0, "the tiles' order holds for every chunk");
constexpr int kSortMax = 16384;  // largest instance reordered (160 KiB of shared memory, 16-bit starts)
constexpr size_t sort_bytes(int cap) { return (size_t)cap * (2 * sizeof(unsigned) + sizeof(uint16_t)); }

}  // namespace

struct BatchState {
    int cap_count = 0;
    int64_t cap_points = 0, cap_tiles = 0;
    void *dev = nullptr;
    size_t dev_bytes = 0;
    BInst *d_table = nullptr;
    Hdr *d_hdr = nullptr;      // the head of a BHdr
    const unsigned *d_first = nullptr;  // and its table
    Rows rows{};               // by row and tile (ev set per launch)
    PackOut pack{};            // the same arrays, writable
    int *d_flags = nullptr, *d_scan = nullptr, *d_part = nullptr;  // by point
    int64_t part_cap = 0;
    int sort_cap = 0;          // instances up to this many points are reordered (a power of two)
    unsigned *d_work = nullptr;
    unsigned *d_status = nullptr;
    int *d_istats = nullptr;
    unsigned long long *d_ev = nullptr;  // pair tests evaluated per instance and pass [count][3]
    unsigned long long *h_ev = nullptr;
    BInst *h_table = nullptr;
    BHdr *h_hdr = nullptr;
    int *h_istats = nullptr;
    unsigned *h_status = nullptr;
    cudaGraphExec_t graph = nullptr;
    int graph_ch = -1, graph_bps = -1, graph_stats = -1;
    int ch = 64, bps = 8;  // column tiles per work item, blocks per SM
    bool tuned = false;
    PhaseMarks marks;  // timing off
};

void batch_release(BatchState *b) {
    if (!b) return;
    if (b->graph) cudaGraphExecDestroy(b->graph);
    if (b->dev) cudaFree(b->dev);
    if (b->h_table) cudaFreeHost(b->h_table);
    if (b->h_hdr) cudaFreeHost(b->h_hdr);
    if (b->h_istats) cudaFreeHost(b->h_istats);
    if (b->h_ev) cudaFreeHost(b->h_ev);
    if (b->h_status) cudaFreeHost(b->h_status);
    delete b;
}

namespace {

size_t al256(size_t v) { return (v + 255) / 256 * 256; }

// (Re)allocates the batch workspace for at least these sizes.
int batch_reserve(BatchState *b, int count, int64_t points, int64_t tiles) {
    if (count <= b->cap_count && points <= b->cap_points && tiles <= b->cap_tiles) return DBSCAN_OK;
    const int nc = std::max(count, b->cap_count);
    const int64_t np = std::max<int64_t>(std::max(points, b->cap_points), 1);
    const int64_t nt = std::max<int64_t>(std::max(tiles, b->cap_tiles), 1), nr = nt * BT;
    const int64_t part = np / 2048 + 4;
    size_t off = 0;
    auto take = [&](size_t bytes) {
        const size_t o = off;
        off = al256(off + bytes);
        return o;
    };
    const size_t o_table = take(sizeof(BInst) * nc), o_hdr = take(sizeof(BHdr)), o_tiles = take(sizeof(TileRec) * nt),
                 o_P16 = take(32 * nr), o_nb = take(4 * nr), o_nbc = take(4 * nr), o_box = take(128 * nt),
                 o_count = take(4 * nr), o_core = take(nr), o_parent = take(4 * nr), o_border = take(4 * nr),
                 o_perm = take(4 * nr), o_least = take(4 * nr), o_tag = take(4 * nt), o_need = take(4 * nt),
                 o_inv = take(4 * np), o_flags = take(4 * np), o_scan = take(4 * (np + 1)), o_part = take(4 * part),
                 o_work = take(4 * 8), o_status = take(16), o_istats = take(16 * nc), o_ev = take(24 * (size_t)nc);
    if (b->graph) {
        cudaGraphExecDestroy(b->graph);
        b->graph = nullptr;
    }
    if (b->dev) cudaFree(b->dev);
    if (b->h_table) cudaFreeHost(b->h_table);
    if (b->h_istats) cudaFreeHost(b->h_istats);
    if (b->h_ev) cudaFreeHost(b->h_ev);
    b->dev = nullptr;
    b->h_table = nullptr;
    b->h_istats = nullptr;
    b->h_ev = nullptr;
    if (cudaMalloc(&b->dev, off) != cudaSuccess) {
        cudaGetLastError();
        b->cap_count = 0;
        b->cap_points = b->cap_tiles = 0;
        return DBSCAN_ERR_OOM;
    }
    if (cudaMallocHost(&b->h_table, sizeof(BInst) * nc) != cudaSuccess ||
        cudaMallocHost(&b->h_istats, 16 * (size_t)nc) != cudaSuccess ||
        cudaMallocHost(&b->h_ev, 24 * (size_t)nc) != cudaSuccess)
        return DBSCAN_ERR_OOM;
    if (!b->h_hdr && cudaMallocHost(&b->h_hdr, sizeof(BHdr)) != cudaSuccess) return DBSCAN_ERR_OOM;
    if (!b->h_status && cudaMallocHost(&b->h_status, 16) != cudaSuccess) return DBSCAN_ERR_OOM;
    char *base = static_cast<char *>(b->dev);
    auto at = [&](size_t o) { return static_cast<void *>(base + o); };
    b->dev_bytes = off;
    b->d_table = static_cast<BInst *>(at(o_table));
    b->d_hdr = static_cast<Hdr *>(at(o_hdr));
    b->d_first = reinterpret_cast<const BHdr *>(b->d_hdr)->first;
    PackOut &w = b->pack;
    w.tiles = static_cast<TileRec *>(at(o_tiles));
    w.perm = static_cast<int *>(at(o_perm));
    w.inv = static_cast<int *>(at(o_inv));
    w.count = static_cast<int *>(at(o_count));
    w.least = static_cast<int *>(at(o_least));
    w.P16 = static_cast<uint2 *>(at(o_P16));
    w.nb = static_cast<float *>(at(o_nb));
    w.box = static_cast<float *>(at(o_box));
    w.cap_tiles = nt;
    Rows &r = b->rows;
    r.tiles = w.tiles;
    r.P16 = w.P16;
    r.nb = w.nb;
    r.nbc = static_cast<float *>(at(o_nbc));
    r.box = w.box;
    r.cap_tiles = nt;
    r.count = w.count;
    r.core = static_cast<uint8_t *>(at(o_core));
    r.parent = static_cast<int *>(at(o_parent));
    r.border = static_cast<int *>(at(o_border));
    r.perm = w.perm;
    r.tag = static_cast<int *>(at(o_tag));
    r.need = static_cast<int *>(at(o_need));
    b->d_flags = static_cast<int *>(at(o_flags));
    b->d_scan = static_cast<int *>(at(o_scan));
    b->d_part = static_cast<int *>(at(o_part));
    b->part_cap = part;
    b->d_work = static_cast<unsigned *>(at(o_work));
    b->d_status = r.status = static_cast<unsigned *>(at(o_status));
    b->d_istats = static_cast<int *>(at(o_istats));
    b->d_ev = static_cast<unsigned long long *>(at(o_ev));
    b->cap_count = nc;
    b->cap_points = np;
    b->cap_tiles = nt;
    if (cudaMemset(b->d_status, 0, 16) != cudaSuccess) return DBSCAN_ERR_CUDA;
    return DBSCAN_OK;
}

// Host table, rows and tiles given out in the order of the passes' queue.
void build_table(const dbscan_instance *inst, int count, const batchitems::Queue &q, BInst *t, int64_t *points,
                 int64_t *tiles, int64_t *max_n) {
    int64_t base = 0, nt = 0, mx = 0;
    for (int k = 0; k < count; ++k) {
        const int i = q.order.empty() ? k : q.order[k];
        const dbscan_instance &in = inst[i];
        BInst &B = t[i];
        B = BInst{};
        const double e = (double)in.eps;
        const int64_t T = (int64_t)std::floor(e * e * 1048576.0);
        const int64_t Tc = std::min<int64_t>(T, (int64_t)in.d * 1023 * 1023);
        B.x = in.points;
        B.labels = in.labels_out;
        TileRec &I = B.rec;
        I.n = (int)in.n;
        I.d = in.d;
        I.Tc = (int)Tc;
        I.Tp1 = (float)(Tc + 1);
        I.min_pts = in.min_pts;
        I.leave = in.min_pts;  // batch outputs labels only
        I.inst = i;
        I.point0 = (int)base;
        I.tile0 = (int)nt;
        I.ntiles = (int)((in.n + BT - 1) / BT);
        base += in.n;
        nt += I.ntiles;
        mx = std::max<int64_t>(mx, in.n);
    }
    *points = base;
    *tiles = nt;
    *max_n = mx;
}

// The pair passes and what lies between them.  SIMT: dot products on the CUDA
// cores (DBSCAN_PREC_EXACT_SIMT).
template <bool SIMT>
void enqueue_passes(BatchState *b, const Rows &R, int ch, int pgrid, int egrid, cudaStream_t st, PhaseMarks &pm) {
    pass_kernel<WT_COUNT, true, SIMT><<<pgrid, NT, 0, st>>>(R, b->d_hdr, ch, b->d_first, b->d_work + 0);
    pm.kernel(SIMT ? "batch_count_simt" : "batch_count", st);
    core_kernel<SIMT><<<egrid, NT, 0, st>>>(R, b->d_hdr);
    pm.kernel(SIMT ? "batch_core_simt" : "batch_core", st);
    pass_kernel<WT_NEAR, true, SIMT><<<pgrid, NT, 0, st>>>(R, b->d_hdr, ch, b->d_first, b->d_work + 1);
    pm.kernel(SIMT ? "batch_union_near_simt" : "batch_union_near", st);
    flatten_kernel<<<egrid, NT, 0, st>>>(R, b->d_hdr);
    pm.kernel("batch_flatten", st);
    pass_kernel<WT_FAR, true, SIMT><<<pgrid, NT, 0, st>>>(R, b->d_hdr, ch, b->d_first, b->d_work + 2);
    pm.kernel(SIMT ? "batch_union_simt" : "batch_union", st);
    pass_kernel<WT_BORDER, true, SIMT><<<pgrid, NT, 0, st>>>(R, b->d_hdr, ch, b->d_first, b->d_work + 3);
    pm.kernel(SIMT ? "batch_border_simt" : "batch_border", st);
}

cudaError_t enqueue_batch(BatchState *b, int label_mode, bool simt, bool stats, int ch, int bps, cudaStream_t st,
                          PhaseMarks *pm = nullptr) {
    PhaseMarks off;
    if (!pm) pm = &off;
    int dev = 0, sms = 148;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const int pgrid = sms * bps, egrid = sms * 8;
    cudaError_t e;
    if ((e = cudaMemcpyAsync(b->d_table, b->h_table, sizeof(BInst) * b->cap_count, cudaMemcpyHostToDevice, st)))
        return e;
    if ((e = cudaMemcpyAsync(b->d_hdr, b->h_hdr, sizeof(BHdr), cudaMemcpyHostToDevice, st))) return e;
    if ((e = cudaMemsetAsync(b->d_work, 0, 4 * 8, st))) return e;
    if (stats && (e = cudaMemsetAsync(b->d_istats, 0, 16 * (size_t)b->cap_count, st))) return e;
    if (stats && (e = cudaMemsetAsync(b->d_ev, 0, 24 * (size_t)b->cap_count, st))) return e;
    Rows R = b->rows;
    R.ev = stats ? b->d_ev : nullptr;
    batch_sortpack_kernel<<<sms * 3, 512, sort_bytes(b->sort_cap), st>>>(b->d_table, b->d_hdr, b->sort_cap, b->pack,
                                                                        b->d_status);
    pm->kernel("batch_prep", st);
    if (simt) enqueue_passes<true>(b, R, ch, pgrid, egrid, st, *pm);
    else enqueue_passes<false>(b, R, ch, pgrid, egrid, st, *pm);
    root_kernel<<<egrid, NT, 0, st>>>(R, b->d_hdr, b->pack.least);
    pm->kernel("batch_root", st);
    const bool compact = label_mode == DBSCAN_LABEL_COMPACT;
    batch_label_kernel<<<egrid, NT, 0, st>>>(R, b->d_hdr, b->d_table, b->pack.inv, b->pack.least,
                                             compact ? b->d_flags : nullptr, stats ? b->d_istats : nullptr);
    pm->kernel("batch_label", st);
    if ((e = cudaGetLastError())) return e;
    if (compact) {
        if ((e = launch_exclusive_scan(b->d_flags, b->d_scan, b->cap_points, b->d_part, b->part_cap, st, pm)))
            return e;
        batch_compact_kernel<<<egrid, 256, 0, st>>>(R, b->d_hdr, b->d_table, b->d_scan);
        pm->kernel("batch_compact", st);
    }
    if (stats && (e = cudaMemcpyAsync(b->h_istats, b->d_istats, 16 * (size_t)b->cap_count, cudaMemcpyDeviceToHost,
                                      st)))
        return e;
    if (stats && (e = cudaMemcpyAsync(b->h_ev, b->d_ev, 24 * (size_t)b->cap_count, cudaMemcpyDeviceToHost, st)))
        return e;
    if ((e = cudaMemcpyAsync(b->h_status, b->d_status, sizeof(unsigned), cudaMemcpyDeviceToHost, st))) return e;
    if ((e = cudaMemsetAsync(b->d_status, 0, sizeof(unsigned), st))) return e;
    return cudaGetLastError();
}

// The whole sequence as one CUDA graph (rebuilt when capacities or the tuned
// configuration change).
int batch_graph_launch(BatchState *b, int label_mode, bool simt, bool stats, cudaStream_t st) {
    if (!b->graph || b->graph_ch != b->ch || b->graph_bps != b->bps ||
        b->graph_stats != (int)stats || b->graph_ch < 0) {
        if (b->graph) {
            cudaGraphExecDestroy(b->graph);
            b->graph = nullptr;
        }
        cudaStream_t cs;
        if (cudaStreamCreateWithFlags(&cs, cudaStreamNonBlocking) != cudaSuccess) return DBSCAN_ERR_CUDA;
        cudaGraph_t g = nullptr;
        cudaError_t e = cudaStreamBeginCapture(cs, cudaStreamCaptureModeThreadLocal);
        if (!e) e = enqueue_batch(b, label_mode, simt, stats, b->ch, b->bps, cs);
        cudaError_t e2 = cudaStreamEndCapture(cs, &g);
        cudaStreamDestroy(cs);
        if (e || e2 || !g) {
            if (g) cudaGraphDestroy(g);
            cudaGetLastError();
            return DBSCAN_ERR_CUDA;
        }
        e = cudaGraphInstantiate(&b->graph, g, 0);
        cudaGraphDestroy(g);
        if (e) {
            cudaGetLastError();
            b->graph = nullptr;
            return DBSCAN_ERR_CUDA;
        }
        b->graph_ch = b->ch;
        b->graph_bps = b->bps;
        b->graph_stats = (int)stats;
    }
    return cudaGraphLaunch(b->graph, st) == cudaSuccess ? DBSCAN_OK : DBSCAN_ERR_CUDA;
}

}  // namespace

namespace {

// One part of a batch, its sizes checked; adds the pair tests per pass to tot.
int batch_run(dbscan_plan *plan, const dbscan_instance *inst, int32_t count, dbscan_stats *per_inst,
              unsigned long long tot[4]) {
    int cur = -1;
    cudaGetDevice(&cur);
    if (cur != plan->opts.device) cudaSetDevice(plan->opts.device);
    if (!plan->batch) plan->batch = new BatchState();
    BatchState *b = plan->batch;
    const int label_mode = plan->opts.label_mode;
    const bool stats = per_inst != nullptr, simt = plan->opts.precision == DBSCAN_PREC_EXACT_SIMT;
    cudaStream_t st = plan->stream;

    std::vector<BInst> tmp(count);
    int64_t points = 0, tiles = 0, max_n = 0;
    const batchitems::Queue queue = batchitems::make_queue(count, [&](int32_t k) { return inst[k].n; });
    if (!queue.fits) return DBSCAN_ERR_UNSUPPORTED;
    build_table(inst, count, queue, tmp.data(), &points, &tiles, &max_n);
    int s = batch_reserve(b, count, points, tiles);
    if (s) return s;
    // Instances up to kSortMax points are put in Z-order; the sort's shared
    // memory is sized for the largest of them.
    int sort_cap = 2;
    while (sort_cap < std::min<int64_t>(max_n, kSortMax)) sort_cap <<= 1;
    if (sort_cap != b->sort_cap && b->graph) {
        cudaGraphExecDestroy(b->graph);
        b->graph = nullptr;
    }
    b->sort_cap = sort_cap;
    if (sort_bytes(sort_cap) > 48 * 1024 &&
        cudaFuncSetAttribute(batch_sortpack_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)sort_bytes(sort_cap)) != cudaSuccess)
        return DBSCAN_ERR_CUDA;

    std::memcpy(b->h_table, tmp.data(), sizeof(BInst) * count);
    if (b->cap_count > count) std::memset(b->h_table + count, 0, sizeof(BInst) * (b->cap_count - count));
    auto prepare = [&](int ch) {
        b->h_hdr->h = Hdr{count, (int)points, (int)tiles,
                          batchitems::step_table(queue, ch / batchitems::kMinChunk, b->h_hdr->first)};
    };

    if (!b->tuned) {
        // Autotune on this batch: every (CH, blocks per SM) candidate, best of 2 runs.
        cudaEvent_t e0, e1;
        cudaEventCreate(&e0);
        cudaEventCreate(&e1);
        float best = 1e30f;
        for (int ch : kCH)
            for (int bps : kBPS) {
                prepare(ch);
                float tbest = 1e30f;
                for (int rep = 0; rep < 2; ++rep) {
                    cudaEventRecord(e0, st);
                    if (enqueue_batch(b, label_mode, simt, false, ch, bps, st)) {
                        cudaEventDestroy(e0);
                        cudaEventDestroy(e1);
                        return DBSCAN_ERR_CUDA;
                    }
                    cudaEventRecord(e1, st);
                    cudaEventSynchronize(e1);
                    float ms = 0.f;
                    cudaEventElapsedTime(&ms, e0, e1);
                    tbest = std::min(tbest, ms);
                }
                if (tbest < best) {
                    best = tbest;
                    b->ch = ch;
                    b->bps = bps;
                }
            }
        cudaEventDestroy(e0);
        cudaEventDestroy(e1);
        b->tuned = true;
    }
    prepare(b->ch);
    if (plan->opts.profile) {  // per-kernel events: run the sequence uncaptured
        plan->marks.begin(st);
        if (enqueue_batch(b, label_mode, simt, stats, b->ch, b->bps, st, &plan->marks)) return DBSCAN_ERR_CUDA;
    } else {
        s = batch_graph_launch(b, label_mode, simt, stats, st);
        if (s) return s;
    }
    if (cudaStreamSynchronize(st) != cudaSuccess) return DBSCAN_ERR_CUDA;
    if (cur >= 0 && cur != plan->opts.device) cudaSetDevice(cur);
    const unsigned bits = *b->h_status;
    if (bits & DB_EBIT_NOT_QUANTISED) return DBSCAN_ERR_NOT_QUANTISED;
    if (bits & DB_EBIT_TIMEOUT) return DBSCAN_ERR_TIMEOUT;
    if (bits) return DBSCAN_ERR_CUDA;
    if (stats) {
        for (int i = 0; i < count; ++i)
            for (int k = 0; k < 3; ++k) tot[k] += b->h_ev[3 * i + k];
        for (int i = 0; i < count; ++i) {
            dbscan_stats &o = per_inst[i];
            std::memset(&o, 0, sizeof(o));
            o.n_core = b->h_istats[4 * i + 0];
            o.n_border = b->h_istats[4 * i + 1];
            o.n_noise = b->h_istats[4 * i + 2];
            o.n_clusters = b->h_istats[4 * i + 3];
            o.candidate_pairs = inst[i].n * inst[i].n;
            o.path = DBSCAN_PATH_ALLPAIRS_SIMT;
            const double e = (double)inst[i].eps;
            o.threshold = (int64_t)std::floor(e * e * 1048576.0);
            o.kernels = 9 + (label_mode == DBSCAN_LABEL_COMPACT ? 4 : 0);
            o.pair_tests = (int64_t)(b->h_ev[3 * i] + b->h_ev[3 * i + 1] + b->h_ev[3 * i + 2]);
        }
    }
    return DBSCAN_OK;
}

}  // namespace

extern "C" int dbscan_batch(dbscan_plan *plan, const dbscan_instance *inst, int32_t count, dbscan_stats *per_inst) {
    if (!plan || count < 0 || (count > 0 && !inst)) return DBSCAN_ERR_ARG;
    if (count == 0) return DBSCAN_OK;
    int64_t total = 0;
    for (int i = 0; i < count; ++i) {
        const dbscan_instance &in = inst[i];
        if (in.n < 0 || in.d < 1 || in.d > 16 || !(in.eps > 0.0f) || std::isinf(in.eps) || in.min_pts < 1)
            return in.d > 16 ? DBSCAN_ERR_UNSUPPORTED : DBSCAN_ERR_ARG;
        if (in.n > 0 && (!in.points || !in.labels_out)) return DBSCAN_ERR_ARG;
        total += in.n;
    }
    if (total > INT32_MAX / 2) return DBSCAN_ERR_ARG;
    // the limit on work: 32-point row tiles x chunks of four 64-point column
    // tiles (about n^2 / 8,192 per instance) in int32
    int64_t items = 0;
    for (int i = 0; i < count; ++i) {
        const int64_t rows = (inst[i].n + 31) / 32, cols = (inst[i].n + 63) / 64;
        items += rows * ((cols + 3) / 4);
    }
    if (items > INT32_MAX) return DBSCAN_ERR_UNSUPPORTED;
    // Rows are counted in int32: a batch of very many tiles runs in parts.  An
    // off-grid instance fails the call, not the instances of the other parts.
    int status = DBSCAN_OK;
    unsigned long long tot[4] = {0, 0, 0, 0};
    for (int32_t i = 0; i < count;) {
        const int32_t end = batchitems::part_end(i, count, [&](int32_t k) { return inst[k].n; });
        const int s = batch_run(plan, inst + i, end - i, per_inst ? per_inst + i : nullptr, tot);
        if (s && s != DBSCAN_ERR_NOT_QUANTISED) return s;
        if (!status) status = s;
        i = end;
    }
    if (status) return status;
    // the batch's pair tests per pass, also left in the plan's counters 16..18
    if (per_inst && cudaMemcpy(plan->w.ctr + DB_CTR_EVAL, tot, sizeof(tot), cudaMemcpyHostToDevice) != cudaSuccess)
        return DBSCAN_ERR_CUDA;
    return DBSCAN_OK;
}

extern "C" int dbscan_batch_config(dbscan_plan *plan, int32_t *chunk_tiles, int32_t *blocks_per_sm) {
    if (!plan) return DBSCAN_ERR_ARG;
    if (!plan->batch || !plan->batch->tuned) return DBSCAN_ERR_NOT_FOUND;
    if (chunk_tiles) *chunk_tiles = plan->batch->ch;
    if (blocks_per_sm) *blocks_per_sm = plan->batch->bps;
    return DBSCAN_OK;
}

extern "C" int dbscan_batch_tile(dbscan_plan *plan, int32_t *tile_rows, int32_t *tile_cols) {
    if (!plan) return DBSCAN_ERR_ARG;
    if (!plan->batch || !plan->batch->tuned) return DBSCAN_ERR_NOT_FOUND;
    if (tile_rows) *tile_rows = BT;
    if (tile_cols) *tile_cols = BT;
    return DBSCAN_OK;
}
