// batch_items.h — how a batch (batch.cu) is cut into parts.  Plain C++, host.
#pragma once

#include <cstdint>

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

}  // namespace batchitems
