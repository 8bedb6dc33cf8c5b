// Check of a group of a sorted sliced layout: its launches address memory by the
// group's descriptor alone.  Plain C++ as well, so that it can be tested without a
// GPU on descriptors that no plan holds.
#pragma once

#include "internal.h"
#include "pieces.h"

namespace spmvk {

// Slices of a group of rows of `len` entries; 1 above the lengths that make groups.
SPMV_HOST_DEVICE int sell_group_size(int len) {
    static_assert(kSellGroupLen == 5, "one case per length");
    constexpr int n0 = kSellGroup[0], n1 = kSellGroup[1], n2 = kSellGroup[2], n3 = kSellGroup[3], n4 = kSellGroup[4];
    switch (len) {
        case 0: return n0;
        case 1: return n1;
        case 2: return n2;
        case 3: return n3;
        case 4: return n4;
        default: return 1;
    }
}

// Whether group i of a rank with groups [g0, g1) and slices [s0, s1) holds the
// slices that follow the group before it: its own fields those of its first
// slice, and, if it is more than a slice, the size for its length, full slices of
// that length with their positions (of npos) and slots one after another.  The
// rank's groups hold all its slices when each of them passes.
SPMV_HOST_DEVICE bool sell_group_ok(const SellSlice* groups, int64_t i, int64_t g0, int64_t g1, const SellSlice* slices,
                                    int64_t s0, int64_t s1, const uint8_t* len, int64_t npos) {
    const SellSlice g = groups[i];
    if (g.group != 1 && g.group != sell_group_size(g.len)) return false;
    const int64_t s = g.first, end = s + g.group;
    if (s < s0 || end > s1 || (i + 1 == g1 && end != s1)) return false;
    if (s != (i == g0 ? s0 : (int64_t)groups[i - 1].first + groups[i - 1].group)) return false;
    for (int k = 0; k < g.group; ++k) {
        const SellSlice d = slices[s + k];
        const int64_t p0 = (int64_t)g.p0 + 32 * k;
        if (d.p0 != p0 || d.off != (int64_t)g.off + 32 * (int64_t)g.len * k || d.len != g.len || d.xoff != g.xoff ||
            d.rows != (k ? 32 : g.rows))
            return false;
        if (g.group == 1) continue;
        if (d.rows != 32 || p0 < 0 || p0 + 32 > npos) return false;
        for (int r = 0; r < 32; ++r)
            if (len[p0 + r] != g.len) return false;
    }
    return true;
}

}  // namespace spmvk
