// tc_items.h — work items of the tensor-core passes (gram_tc.cu): how many there
// are, and the row unit and column chunk of each.  Plain C++, for the host and
// the device.
#pragma once

#include <cstdint>

#ifndef DB_HD
#ifdef __CUDACC__
#define DB_HD __host__ __device__ __forceinline__
#else
#define DB_HD inline
#endif
#endif

namespace tcitems {

// Column tiles per work item: about 8 items per SM, a power of two up to 16
// (an item of 16 tiles keeps an SM busy for some 20 us, the longest tail).
inline int chunk_tiles(int64_t units, int64_t nct, int sms) {
    int c = 16;
    while (c > 1 && units * ((nct + c - 1) / c) < (int64_t)8 * sms) c >>= 1;
    return c;
}

// Items of a pass over `units` row units and `rels` chunks each.  64 bits: at
// 2^25 points, units of 128 rows and chunks of 16 tiles make 2^31 items, and a
// verification takes any number of points.
DB_HD int64_t count(int units, int rels) { return (int64_t)units * rels; }

// Item w: its row unit, and its chunk (counted from the unit's own, or from the
// first); the chunks nearest the units' own come first for all units.
struct Item {
    int unit, rel;
};
DB_HD Item item(int64_t w, int units) {
    const int64_t rel = w / units;
    return {(int)(w - rel * units), (int)rel};
}

// First item of CTA `cta` when the items are dealt out 32 at a time, a lane
// each: lane l of the round from `base` looks at item base + l * ctas, and the
// next round starts at base + round(ctas).
DB_HD int64_t dealt(int64_t base, int lane, int ctas) { return base + (int64_t)lane * ctas; }
DB_HD int64_t round(int ctas) { return (int64_t)ctas * 32; }

}  // namespace tcitems
