// skip_shape.h -- offsets into the rectangle tables that the skip boxes are built
// from (skip.cu): kSkipLevels^2 tables, one per rectangle size, of a word per
// column of bricks (with kSkipPad columns before the grid) and 64 layers.
#pragma once

#ifdef __CUDACC__
#define SALF_HD __host__ __device__ __forceinline__
#else
#define SALF_HD inline
#endif

constexpr int kSkipLevels = 5;  // rectangles of 1, 2, 4, 8, 16 columns a side
constexpr int kSkipPad = (1 << (kSkipLevels - 1)) - 1;  // they may start this far before the grid

// From a column's word in the first table to the word of the 2^i x 2^j rectangle
// dx, dy columns away, `table` words per table, px a row.
template <class Off>
SALF_HD Off skip_rect_offset(int i, int j, Off table, int px, int dy, int dx) {
  return (Off)(i * kSkipLevels + j) * table + ((Off)dy * px + dx);
}

// Whether offsets into all the tables need 64 bits.  A grid of 64 layers or more
// has at most 2^26 words per table (2^28 bricks, narrow grids and their padding
// included); a flat one has a word for each of up to 2^28 columns, and 24 tables
// pass 2^31 from 89M on (40000 x 40000 x 4 cells: 100M).  32 bits are the faster
// ones (k_skip_boxes on 1.27M voxels, 158 us instead of 193).
inline bool skip_wide_offsets(long long table) {
  return table * (kSkipLevels * kSkipLevels) > 0x7fffffffLL;
}
