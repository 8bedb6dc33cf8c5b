// Pieces of a long row of the batched products: piece p of a row of `len`
// entries holds the entries [p piece_len, (p + 1) piece_len) of the row that
// exist.  Counted within the row: a matrix may have up to 2^31 - 9 entries, so
// an entry index plus a piece length can pass 2^31.  Plain C++ as well, so that
// the arithmetic can be tested without a GPU.
#pragma once

#ifdef __CUDACC__
#define SPMV_HOST_DEVICE __host__ __device__ __forceinline__
#else
#define SPMV_HOST_DEVICE inline
#endif

namespace spmvk {

SPMV_HOST_DEVICE int piece_count(int len, int piece_len) { return len / piece_len + (len % piece_len != 0); }

// Entries of piece p < piece_count(len, piece_len).
SPMV_HOST_DEVICE int piece_size(int len, int piece_len, int p) {
    const int left = len - p * piece_len;
    return left < piece_len ? left : piece_len;
}

}  // namespace spmvk
