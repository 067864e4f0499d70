// pairs_wt.cu — one instance's all-pairs run for d <= 16 on the warp tiles
// (warp_tile.cuh): the default where no grid applies (9 <= d <= 15, d = 16 below
// the tensor-core path's size, eps too large for the projected grid, grid off).
//
// The points are put in Z-order of all their coordinates by a counting sort:
// the top bits of every axis, as many as make about 2 n cells (at most 2^18).
// Groups then differ in some bit of some axis, and tiles are mostly of one
// group.  Count, core flags, merge and border run as in the batch.
// 30,011 points in 15 groups plus 15% noise, d = 12: 2.87 ms with 64 x 64 FP32
// tiles in index order (1.4e9 pair tests, each d + 2 FP32 operations); on warp
// tiles in Z-order of three coordinates 0.52 ms, where 35% of the tiles hold core
// points of several groups and the merge has to test 14% of the tile pairs;
// 0.37 ms with all axes' bits (6% of the tiles, 6% of the pairs).
#include <algorithm>

#include "warp_tile.cuh"

using namespace wtile;

namespace {

// Z-order code over d axes: the first `total` bits, highest bits of all axes
// first (total <= 10 d).
__global__ void __launch_bounds__(256) wt_code_kernel(const float *__restrict__ x, int n, int d, int total,
                                                      int *__restrict__ code, int *__restrict__ rank, int *hist) {
    db::wait_prior_grid();  // started as a programmatic dependent
    db::allow_next_grid();
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const float *p = x + (size_t)i * d;
    int c = 0;
    for (int left = total, bit = 9; left > 0; --bit)
        for (int j = 0; j < d && left > 0; ++j, --left) {
            int u;
            db::on_grid(p[j], u);  // off-grid input is reported when the row is packed
            c = 2 * c | (u >> bit & 1);
        }
    code[i] = c;
    rank[i] = atomicAdd(hist + c, 1);
}

__global__ void __launch_bounds__(256) wt_scatter_kernel(int n, const int *__restrict__ code,
                                                         const int *__restrict__ rank, const int *__restrict__ start,
                                                         int *__restrict__ order) {
    db::wait_prior_grid();
    db::allow_next_grid();
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) order[start[code[i]] + rank[i]] = i;
}

__global__ void __launch_bounds__(256) wt_pack_kernel(const float *__restrict__ x, TileRec I,
                                                      const int *__restrict__ order, PackOut w, Hdr h, Hdr *hdr,
                                                      unsigned *work, unsigned *status) {
    db::wait_prior_grid();
    db::allow_next_grid();
    const int T = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5);
    if (blockIdx.x == 0 && threadIdx.x < 4) work[threadIdx.x] = 0u;
    if (blockIdx.x == 0 && threadIdx.x == 0) *hdr = h;
    if (T >= I.ntiles) return;
    if (pack_tile_d(x, I, T, order, w)) atomicOr(status, DB_EBIT_NOT_QUANTISED);
}

// Labels (a core point: the smallest point index of its set; a border point:
// that of its smallest-index core neighbour; noise: -1), the optional counts
// and core flags, and the run's statistics.
__global__ void __launch_bounds__(256) wt_label_kernel(Rows R, int n, const int *__restrict__ inv,
                                                       const int *__restrict__ least, int *__restrict__ labels,
                                                       int *__restrict__ counts_out, uint8_t *__restrict__ core_out,
                                                       unsigned long long *ctr, unsigned *status_out) {
    db::wait_prior_grid();
    db::allow_next_grid();
    db::report_status(R.status, status_out);
    __shared__ int red[4];
    if (threadIdx.x < 4) red[threadIdx.x] = 0;
    __syncthreads();
    const int g = blockIdx.x * blockDim.x + threadIdx.x;
    int kind = -1;
    bool root = false;
    if (g < n) {
        const int o = R.perm[g], bo = R.border[g];
        int lab = -1;
        kind = 2;
        if (R.core[g]) {
            const int r = R.parent[g];
            lab = least[r];
            root = r == g;
            kind = 0;
        } else if (bo != DB_NONE) {
            lab = least[R.parent[inv[bo]]];
            kind = 1;
        }
        labels[o] = lab;
        if (counts_out) counts_out[o] = R.count[g];
        if (core_out) core_out[o] = kind == 0;
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const unsigned m = __ballot_sync(FULL, k < 3 ? kind == k : root);
        if ((threadIdx.x & 31) == 0 && m) atomicAdd(&red[k], __popc(m));
    }
    __syncthreads();
    if (threadIdx.x < 4 && red[threadIdx.x]) atomicAdd(ctr + 2 + threadIdx.x, (unsigned long long)red[threadIdx.x]);
}

// Bits of the counting sort's cells: about 2 n cells, at most 2^kWtMaxCellBits.
int cell_bits(int64_t n) {
    int lg = 1;
    while ((int64_t(1) << lg) < n) ++lg;
    return std::min(lg + 1, kWtMaxCellBits);
}

}  // namespace

size_t wt_bytes(int64_t n) {
    const size_t nt = (size_t)((n + BT - 1) / BT), nr = nt * BT;
    auto al = [](size_t v) { return (v + 255) / 256 * 256; };
    return al(nt * sizeof(TileRec)) + al(nr * 32) + 8 * al(nr * 4) + al(nr) + al(nt * 128) + 2 * al(nt * 4) +
           al((size_t)n * 4) + al((size_t)4 << cell_bits(n)) + 512;
}

cudaError_t launch_allpairs_wt(const DbWork &w, const float *x, int64_t n64, int32_t d, int64_t Tc, int32_t min_pts,
                               bool exact, int32_t *labels, int32_t *counts_out, uint8_t *core_out, cudaStream_t st) {
    const int n = (int)n64, nt = (n + BT - 1) / BT, nr = nt * BT;
    char *at = static_cast<char *>(w.wt);
    auto take = [&](size_t bytes) {
        char *p = at;
        at += (bytes + 255) / 256 * 256;
        return static_cast<void *>(p);
    };
    PackOut o{};
    o.tiles = static_cast<TileRec *>(take(nt * sizeof(TileRec)));
    o.P16 = static_cast<uint2 *>(take((size_t)nr * 32));
    o.nb = static_cast<float *>(take((size_t)nr * 4));
    Rows R{};
    R.nbc = static_cast<float *>(take((size_t)nr * 4));
    o.count = static_cast<int *>(take((size_t)nr * 4));
    R.parent = static_cast<int *>(take((size_t)nr * 4));
    R.border = static_cast<int *>(take((size_t)nr * 4));
    o.perm = static_cast<int *>(take((size_t)nr * 4));
    o.least = static_cast<int *>(take((size_t)nr * 4));
    int *order = static_cast<int *>(take((size_t)nr * 4));
    R.core = static_cast<uint8_t *>(take(nr));
    o.box = static_cast<float *>(take((size_t)nt * 128));
    R.tag = static_cast<int *>(take((size_t)nt * 4));
    R.need = static_cast<int *>(take((size_t)nt * 4));
    o.inv = static_cast<int *>(take((size_t)n * 4));
    int *hist = static_cast<int *>(take((size_t)4 << cell_bits(n)));
    unsigned *work = static_cast<unsigned *>(take(64));
    Hdr *hdr = static_cast<Hdr *>(take(sizeof(Hdr)));
    o.cap_tiles = nt;
    R.tiles = o.tiles;
    R.P16 = o.P16;
    R.nb = o.nb;
    R.box = o.box;
    R.cap_tiles = nt;
    R.count = o.count;
    R.perm = o.perm;
    R.status = w.status;
    R.ev = w.ctr + DB_CTR_EVAL;
    TileRec I{};
    I.ntiles = nt;
    I.n = n;
    I.d = d;
    I.Tc = (int)Tc;
    I.Tp1 = (float)(Tc + 1);
    I.min_pts = min_pts;
    I.leave = exact ? INT_MAX : min_pts;
    // column tiles per work item (2^19 tiles of 2,048 chunks at most: 32 bits hold
    // two items each): enough items (two a tile and chunk) to fill the
    // chip some four times over, 8 to 256 tiles each
    int ch = 256;
    while (ch > 8 && 2 * (int64_t)nt * ((nt + ch - 1) / ch) < 16384) ch >>= 1;
    const Hdr h{1, n, nt, (nt + ch - 1) / ch};

    cudaError_t e;
    int *code = R.parent, *rank = R.border;  // free until the core kernel
    const int total = std::min(cell_bits(n), 10 * d), cells = 1 << total;
    if ((e = cudaMemsetAsync(hist, 0, sizeof(int) * (size_t)cells, st))) return e;
    const int nb = (n + 255) / 256;
    launch_dependent(wt_code_kernel, nb, 256, st, x, n, d, total, code, rank, hist);
    w.marks->kernel("wt_code", st);
    if ((e = launch_bucket_scan(hist, cells, st))) return e;
    w.marks->kernel("wt_scan", st);
    launch_dependent(wt_scatter_kernel, nb, 256, st, n, code, rank, hist, order);
    w.marks->kernel("wt_scatter", st);
    launch_dependent(wt_pack_kernel, (nt + 7) / 8, 256, st, x, I, order, o, h, hdr, work, w.status);
    w.marks->kernel("wt_pack", st);
    const int grid = 152 * 3, tgrid = std::min((nt + 7) / 8, 152 * 8);
    launch_dependent(pass_kernel<WT_COUNT, false, false>, grid, NT, st, R, hdr, ch, nullptr, work);
    w.marks->kernel("wt_count", st);
    launch_dependent(core_kernel<false>, std::min(tgrid, 152 * 3), NT, st, R, hdr);
    w.marks->kernel("wt_core", st);
    launch_dependent(pass_kernel<WT_NEAR, false, false>, std::min((2 * nt + 7) / 8, grid), NT, st, R, hdr, ch, nullptr, work + 1);
    w.marks->kernel("wt_union_near", st);
    launch_dependent(flatten_kernel, tgrid, NT, st, R, hdr);
    w.marks->kernel("wt_flatten", st);
    launch_dependent(pass_kernel<WT_FAR, false, false>, grid, NT, st, R, hdr, ch, nullptr, work + 2);
    w.marks->kernel("wt_union", st);
    launch_dependent(pass_kernel<WT_BORDER, false, false>, grid, NT, st, R, hdr, ch, nullptr, work + 3);
    w.marks->kernel("wt_border", st);
    launch_dependent(root_kernel, std::min(nr / 64, 152 * 8), NT, st, R, hdr, o.least);
    w.marks->kernel("wt_root", st);
    launch_dependent(wt_label_kernel, nb, 256, st, R, n, o.inv, o.least, labels, counts_out, core_out, w.ctr,
                     w.status_out);
    w.marks->kernel("labels", st);
    return cudaGetLastError();
}
