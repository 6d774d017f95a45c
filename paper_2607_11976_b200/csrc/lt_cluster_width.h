// How many CTAs share a row or a group: rules on sizes alone, apart from the kernels so that they can be tested without a GPU.
#pragma once

namespace lt {

constexpr int kSelDirect = 16384;  // rows up to this length are selected by one CTA (a few batches of registers)

// CTAs that share a row of n_keys > kSelDirect keys: as many as the row is long, no more than `widest`, the widest cluster the device
// can place.  Clusters of 16 need a whole GPC, and are asked for only while few are wanted.
inline int select_cluster_width(int n_keys, int n_rows, int widest) {
  int width = 2;
  while (width < 16 && static_cast<long long>(width) * kSelDirect < n_keys) width <<= 1;
  if (width > 8 && static_cast<long long>(n_rows) * width > 128) width = 8;
  return width < widest ? width : widest;
}

}  // namespace lt
