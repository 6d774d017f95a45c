// How a scan is cut into work items and dealt to its CTAs: arithmetic on sizes alone, apart from the kernels so that it can be tested
// without a GPU.
#pragma once

#if defined(__CUDACC__)
#define LT_HOST_DEVICE __host__ __device__ __forceinline__
#else
#define LT_HOST_DEVICE inline
#endif

namespace lt {

// Key tiles to an item, as asked for: more than there are means all of them.
inline int clamp_segment(int seg_tiles, int n_tiles) { return seg_tiles < n_tiles ? seg_tiles : n_tiles; }

// Items are (key segment, query block) pairs, segment-major.  The numbers are unsigned: those of the last round go up to a grid's width
// past the last item.
LT_HOST_DEVICE unsigned int count_items(int n_tiles, int seg_tiles, int n_blocks) {
  const unsigned int seg = static_cast<unsigned int>(seg_tiles);
  return static_cast<unsigned int>(n_blocks) * ((static_cast<unsigned int>(n_tiles) + seg - 1u) / seg);
}
LT_HOST_DEVICE unsigned int count_rounds(unsigned int n_items, unsigned int grid) { return n_items / grid + (n_items % grid != 0u ? 1u : 0u); }

// Dealt out to and fro (CTA 0 .. G - 1, then G - 1 .. 0): the CTA with the longest item of a round gets the shortest of the next.
LT_HOST_DEVICE unsigned int item_of_round(unsigned int round, unsigned int cta, unsigned int grid) {
  return round * grid + ((round & 1u) != 0u ? grid - 1u - cta : cta);
}

// The item's query block (within a segment the last come first) and its first key tile; false for numbers past the last item.
LT_HOST_DEVICE bool split_item(unsigned int item, unsigned int n_items, int n_blocks, int seg_tiles, int& block, int& tile_lo) {
  if (item >= n_items) return false;
  const unsigned int seg = item / static_cast<unsigned int>(n_blocks);
  block = n_blocks - 1 - static_cast<int>(item - seg * static_cast<unsigned int>(n_blocks));
  tile_lo = static_cast<int>(seg) * seg_tiles;
  return true;
}

}  // namespace lt
