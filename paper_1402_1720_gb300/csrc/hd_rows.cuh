// Rows of the hull-restricted system matrix, a chunk of n histories (at most
// kRowsChunk) at a time: the walks of its paths (kPathWords words each), the
// row lengths (row_ptr[i + 1] = row length, and row_ptr[0] = 0 for the first
// chunk; row_ptr points at the chunk's first entry), in-place inclusive scan of
// row_ptr[1..n] over all histories (scratch of rows_scan_scratch(n) int64), and
// the rows into cols at row_ptr[i].  counters: two words the passes of a chunk
// hand its paths out by (launch_rows_count clears both).  The hull is packed (rows_hull_words(V)
// words and one of padding, voxel v at bit v & 31 of word v >> 5).
#pragma once

#include "hd_internal.cuh"

namespace hd {

constexpr int64_t kRowsChunk = int64_t(1) << 22;  // 268 MB of walks
constexpr int64_t kRowsLeast = int64_t(1) << 10;  // 64 KB

// Walks to allocate for calls of n histories: a chunk's when there is room, else
// half as many, and so on (more chunks, each set up once more for the second pass).
// try_alloc(walks) allocates; 0 when not even kRowsLeast of them fit.
template <class TryAlloc>
int64_t rows_walks_room(int64_t n, TryAlloc try_alloc)
{
    int64_t walks = n < kRowsChunk ? n : kRowsChunk;
    while (!try_alloc(walks)) {
        if (walks <= kRowsLeast) return 0;
        walks = walks / 2 > kRowsLeast ? walks / 2 : kRowsLeast;
    }
    return walks;
}

int64_t rows_hull_words(int64_t V);
cudaError_t launch_rows_setup(const Inputs &in, int64_t n, const GeomQ &g, const Cordic &cd,
                              uint32_t *walks, int sm_count, cudaStream_t s);
cudaError_t launch_rows_count(const uint32_t *walks, int64_t n, const GeomQ &g,
                              const uint32_t *hull_bits, unsigned *counters, int64_t *row_ptr,
                              bool first, int sm_count, cudaStream_t s);
int64_t rows_scan_scratch(int64_t n);
cudaError_t launch_rows_scan(int64_t *a, int64_t n, int64_t *scratch, cudaStream_t s);
cudaError_t launch_rows_emit(const uint32_t *walks, int64_t n, const GeomQ &g,
                             const uint32_t *hull_bits, unsigned *counters, const int64_t *row_ptr,
                             int32_t *cols, int sm_count, cudaStream_t s);

}  // namespace hd
