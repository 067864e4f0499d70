// batch_items.h — how a batch (batch.cu) is cut into parts and a part's work is
// numbered.  Plain C++, for the host and (seek) the device.
#pragma once

#include <algorithm>
#include <cstdint>
#include <vector>

#ifndef DB_HD
#ifdef __CUDACC__
#define DB_HD __host__ __device__ __forceinline__
#else
#define DB_HD inline
#endif
#endif

namespace batchitems {

constexpr int kTileRows = 64;  // rows of a tile (warp_tile.cuh)

inline int64_t tiles_of(int64_t n) { return (n + kTileRows - 1) / kTileRows; }

// Tiles of one part.  Rows are counted in int32, and the kernels that stride
// over them add one grid's threads to the last row (with as many rows as an int
// holds, that sum wrapped), so 2^31 / 64 tiles are too many.  2^20 also bound
// the workspace: every instance takes whole tiles of some 4 KB, so ten million
// instances of a few points would ask for 40 GB in one part, and a part this
// long fills the chip for tens of milliseconds as it is.
constexpr int64_t kPartTiles = int64_t(1) << 20;

// End of the part that starts at instance `from`; size_of(i) is the number of
// points of instance i.  At least one instance.
template <typename Size>
int32_t part_end(int32_t from, int32_t count, Size size_of) {
    int64_t tiles = 0;
    int32_t end = from;
    while (end < count && (end == from || tiles + tiles_of(size_of(end)) <= kPartTiles)) tiles += tiles_of(size_of(end++));
    return end;
}

// ---- the queue of a pass ----
// A pass visits every tile with every column chunk of its instance, two work
// items each (the tile's halves).  Step s takes the tiles of all instances that
// have more than s chunks, each with the chunk s after its own, so the tiles
// around the diagonal come first.  Tiles lie in descending order of their
// instances' chunks, so a step's tiles are the first ones, and the queue is the
// steps one after the other: first[s] tiles before step s, and no item that has
// nothing to do.  With as many steps for every tile as the largest instance has,
// 300,000 points beside a million instances of 64 took 142 ms (all warps claiming
// 1.5e8 items a pass from one address, for 2.7e6 that there are), so 94; 4,096
// instances of 64 to 8,192 points 4.22 and 4.10 ms.

constexpr int kMinChunk = 64;    // the smallest column chunk (tiles) a pass is run with
constexpr int kMaxSteps = 1024;  // chunks of the largest instance a batch takes (65,536 tiles)
// 32 bits hold a part's queue, two items an entry, and what is claimed past its end
static_assert(2 * kPartTiles * kMaxSteps <= int64_t(1) << 31, "entries of a part");

inline int64_t steps_of(int64_t tiles, int chunk) { return (tiles + chunk - 1) / chunk; }

struct Queue {
    std::vector<int32_t> order;  // instances in descending order of their chunks (empty: as they are)
    unsigned tiles[kMaxSteps + 1] = {};  // tiles of the instances of k chunks of kMinChunk tiles
    bool fits = true;            // false: an instance has more than kMaxSteps chunks
};

// The order (a counting sort; equal instances keep theirs, and so it holds for
// multiples of kMinChunk too) and the tiles of a part's instances.
template <typename Size>
Queue make_queue(int32_t count, Size size_of) {
    Queue q;
    std::vector<int32_t> at(kMaxSteps + 2, 0);
    bool ascends = false;
    for (int32_t i = 0; i < count;) {  // by runs of instances with as many chunks
        const int64_t k = steps_of(tiles_of(size_of(i)), kMinChunk);
        if (k > kMaxSteps) {
            q.fits = false;
            return q;
        }
        const int32_t i0 = i;
        unsigned t = 0;
        for (int64_t m; i < count && steps_of(m = tiles_of(size_of(i)), kMinChunk) == k; ++i) t += (unsigned)m;
        q.tiles[k] += t;
        at[kMaxSteps - k + 1] += i - i0;
        ascends |= i < count && steps_of(tiles_of(size_of(i)), kMinChunk) > k;
    }
    if (!ascends) return q;
    for (int k = 0; k <= kMaxSteps; ++k) at[k + 1] += at[k];
    q.order.resize(count);
    for (int32_t i = 0; i < count; ++i) q.order[at[kMaxSteps - steps_of(tiles_of(size_of(i)), kMinChunk)]++] = i;
    return q;
}

// first[0 .. steps] for column chunks of m x kMinChunk tiles; returns the steps.
// first[1] is set in any case.
inline int step_table(const Queue &q, int m, unsigned *first) {
    unsigned in = 0;  // tiles of the step
    int steps = 0;
    for (int k = 1; k <= kMaxSteps; ++k) {
        in += q.tiles[k];
        if (q.tiles[k]) steps = (k + m - 1) / m;
    }
    first[0] = first[1] = 0;
    for (int s = 0, k = 1; s < steps; ++s) {
        first[s + 1] = first[s] + in;
        for (; k <= kMaxSteps && k <= (s + 1) * m; ++k) in -= q.tiles[k];  // theirs end with this step
    }
    return steps;
}

// The step of entry w of the queue, from an earlier entry's step on.
DB_HD int step_at(unsigned w, int step, const unsigned *first) {
    while (w >= first[step + 1]) ++step;
    return step;
}

}  // namespace batchitems
