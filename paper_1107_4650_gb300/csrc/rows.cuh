// The rows of a segment, counted from its first one in 32 bits; the grid has nr < 2^31 of them.
#pragma once

#include <stdint.h>
#ifdef __CUDACC__
#include <cuda_runtime.h>
#define DIRAC_ROWS_HD __host__ __device__ __forceinline__
#else
#define DIRAC_ROWS_HD static inline
#endif

namespace dirac {

constexpr int64_t kMaxSegRows = 1 << 30;  // of a segment
struct SegRows {
    int64_t row0;  // the segment's first row in the grid's numbering
    int end, top;  // [0, end) are the segment's; top: the grid's end, or some row far beyond the segment's halo
};
DIRAC_ROWS_HD SegRows seg_rows(int64_t seg, int64_t seg_h, int64_t nr) {
    const int64_t row0 = seg * seg_h, left = nr - row0;
    return {row0, (int)(seg_h < left ? seg_h : left), (int)(left < 2 * kMaxSegRows - 1 ? left : 2 * kMaxSegRows - 1)};
}

// Row r of a segment, a few rows beyond either end, in the grid's numbering modulo 2^32: rows before the grid's first are 2^32
// less a few.
DIRAC_ROWS_HD bool row_in_grid(uint32_t row0, int r, uint32_t nr) { return row0 + (uint32_t)r < nr; }
// and wrapped (periodic grids)
DIRAC_ROWS_HD uint32_t wrap_row(uint32_t row0, int r, uint32_t nr) {
    uint32_t g = row0 + (uint32_t)r;
    while (g > 0xffffff00u) g += nr;
    while (g >= nr) g -= nr;
    return g;
}

}  // namespace dirac
