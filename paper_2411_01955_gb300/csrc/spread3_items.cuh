// Work items of the volume plans' tile-owned spreading, from the number of list entries of
// every tile (host code, no CUDA calls).
#pragma once

#include <cstdint>
#include <vector>

#include <vector_functions.h>

struct Spread3Items {
    std::vector<int64_t> first;   // [tiles] first entry of a tile's list: all lists may pass 2^31 entries
    std::vector<int4> items;      // (tile, first entry, end entry, partial slot or -1), entries within the tile's list
    std::vector<int2> tinfo;      // [tiles] (items, first partial slot or -1)
    int64_t entries = 0;
    int slots = 0;                // partial tiles: one for each item of a tile that has several
};

// Every tile's entries in pieces of at most `item`, an empty tile one empty item.
inline Spread3Items spread3_items(const std::vector<int>& counts, int64_t item) {
    Spread3Items out;
    out.first.resize(counts.size());
    out.tinfo.resize(counts.size());
    for (size_t t = 0; t < counts.size(); ++t) {
        const int64_t n = counts[t];
        const int k = n > item ? (int)((n + item - 1) / item) : 1;
        out.first[t] = out.entries;
        out.tinfo[t] = make_int2(k, k > 1 ? out.slots : -1);
        for (int i = 0; i < k; ++i)
            out.items.push_back(make_int4((int)t, (int)(n * i / k), (int)(n * (i + 1) / k), k > 1 ? out.slots + i : -1));
        if (k > 1) out.slots += k;
        out.entries += n;
    }
    return out;
}

// The same with the smallest pieces, item or more by powers of two, whose partial tiles are
// at most max_slots (pieces of a whole tile need none).
inline Spread3Items spread3_items_within(const std::vector<int>& counts, int64_t item, int64_t max_slots) {
    Spread3Items out = spread3_items(counts, item);
    while (out.slots > max_slots) out = spread3_items(counts, item *= 2);
    return out;
}
