// Chunks that a warp of the merge-path product walks its entries in: 32 lanes of
// MERGE_LANE consecutive entries, from a multiple of MERGE_LANE on.  Unsigned: a
// plan may have up to 2^31 - 65 entries, and the last chunk may end past 2^31.
// Plain C++ as well, so that the walk can be tested without a GPU.
#pragma once

#include "pieces.h"

namespace spmvk {

constexpr int MERGE_LANE = 8;                 // entries per lane and chunk
constexpr int MERGE_CHUNK = 32 * MERGE_LANE;  // entries per chunk

SPMV_HOST_DEVICE unsigned merge_first_chunk(int k0) { return (unsigned)k0 & ~(unsigned)(MERGE_LANE - 1); }

// Whether entry e of a chunk lies in the range [k0, k1).
SPMV_HOST_DEVICE bool merge_in_range(unsigned e, int k0, int k1) { return e >= (unsigned)k0 && e < (unsigned)k1; }

// Whether a row that ends before entry `end` ends in the chunk at c or before it.
SPMV_HOST_DEVICE bool merge_ends_by(int end, unsigned c) { return (unsigned)end <= c + MERGE_CHUNK; }

}  // namespace spmvk
