// grid_dev.cuh — device helpers of the eps-grid paths (grid.cu, grid_rows.cu).
#pragma once

#include "internal.cuh"

namespace {

constexpr unsigned FULL = 0xffffffffu;

// Exact score T + 1 - D(p,q) in the Gram form of Section IV-B: every partial
// sum is an integer below 2*3*1023^2 < 2^24 in magnitude, so FP32 is exact.
template <int D>
__device__ __forceinline__ bool is_nbr(float cp, float px2, float py2, float pz2, float4 q) {
    float acc = cp + q.w;
    acc = fmaf(px2, q.x, acc);
    if (D > 1) acc = fmaf(py2, q.y, acc);
    if (D > 2) acc = fmaf(pz2, q.z, acc);
    return acc >= 1.f;
}

// A point whose neighbour cells hold at most this many points walks them in
// its own thread; the points of a cell with more are walked by the whole warp,
// 32 candidates a step (a cell next to a tight blob can hold thousands).
constexpr int kThreadWalkMax = 96;

// ---- warp-cooperative candidate walk ---------------------------------------
// The neighbour list of a cell is read 32 entries at a time: lane l holds
// (start, size) of one neighbour cell and an inclusive prefix of the sizes, so
// the candidates of those cells form one flattened range that the 32 lanes
// walk together.

__device__ __forceinline__ int warp_incl_scan(int v) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        int y = __shfl_up_sync(FULL, v, o);
        if (lane >= o) v += y;
    }
    return v;
}

// Lane k holding flattened candidate j: the smallest lane with incl[k] > j (a
// 5-step binary search over the lanes' prefixes); its position is then
// start[k] + (j - exclusive[k]).  All 32 lanes must call it; the result is
// meaningless when j >= total.
__device__ __forceinline__ int locate_lane(int j, int incl) {
    int k = 0;
#pragma unroll
    for (int step = 16; step >= 1; step >>= 1)
        if (__shfl_sync(FULL, incl, k + step - 1) <= j) k += step;
    return k & 31;
}

// A point of the grid as {u0, u1, u2, -|u|^2} from its packed form
// u0 | u1 << 10 | u2 << 20 (low 30 bits of a cell_mid entry).
__device__ __forceinline__ float4 unpack_point(unsigned long long key) {
    const unsigned v = (unsigned)key;
    const float x = (float)(v & 1023u), y = (float)((v >> 10) & 1023u), z = (float)((v >> 20) & 1023u);
    return make_float4(x, y, z, -(x * x + y * y + z * z));
}

// Segmented minimum over a warp whose lanes hold consecutive grouped
// positions (so equal cell ids are contiguous): afterwards the first lane of
// each run of equal `cell` holds the minimum of `v` over its run.
template <typename V>
__device__ __forceinline__ V seg_min_down(V v, int cell) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const V y = __shfl_down_sync(FULL, v, o);
        const int cy = __shfl_down_sync(FULL, cell, o);
        if (lane + o < 32 && cy == cell) v = y < v ? y : v;
    }
    return v;
}

}  // namespace
