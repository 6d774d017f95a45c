// How many CTAs share a row or a group: rules on sizes alone, apart from the kernels so that they can be tested without a GPU.
#pragma once

namespace lt {

constexpr int kSelDirect = 16384;  // rows up to this length are selected by one CTA (a few batches of registers)

// CTAs that share a row of n_keys > kSelDirect keys: as many as the row is long, no more than `widest`, the widest cluster the device
// can place.  While few CTAs are wanted a share is half as long (1 x 20 K keys, whole call, width 2 / 4: 18.1 / 16.7 us; 7 x 40 K, 4 / 8: 24.0 /
// 22.9), but not beyond clusters of 8 (1 x 128 K, 8 / 16: 22.2 / 22.6).  Clusters of 16 need a whole GPC, and are asked for only while few are wanted.
constexpr int kSelFewCtas = 32;
inline int select_cluster_width(int n_keys, int n_rows, int widest) {
  int width = 2;
  auto share = [&](int w) { return w < 8 && static_cast<long long>(n_rows) * w <= kSelFewCtas ? kSelDirect / 2 : kSelDirect; };
  while (width < 16 && static_cast<long long>(width) * share(width) < n_keys) width <<= 1;
  if (width > 8 && static_cast<long long>(n_rows) * width > 128) width = 8;
  return width < widest ? width : widest;
}

// CTAs that share one group of the union of n_groups groups of `rows` rows with at most `entries` selected positions each.
// at_once(w): clusters of w CTAs that run at the same time; a second wave pays the clearing, combining and sweeping of its copies of
// the bitmap all over (1024 rows x 512 over 262,144 positions in 64 groups, width 2 / 4 / 8: 16 / 22 / 38 us).  Each doubling
// halves the entries of a CTA and adds copies.  As long as every CTA has an SM to itself that pays down to kUnionFewEntries
// entries (1024 x 32 over 2^20 positions in 16 groups, width 1 / 2 / 4: 22 / 21 / 20 us); CTAs that share an SM have to have
// kUnionManyEntries or more to share out (4096 x 2048 over 131,072 positions in 64 groups, width 2 / 4 / 8: 93 / 66 / 63 us; but 500 x 1024 in
// 125 groups, 1 / 2 / 4: 12 / 17 / 22 us).  Clusters of 16 need a whole GPC: only for few groups.
constexpr long long kUnionFewEntries = 256;
constexpr long long kUnionManyEntries = 16384;
template <class AtOnce>
inline int union_cluster_width(int n_groups, int rows, long long entries, int sms, AtOnce&& at_once) {
  int width = 1;
  while (width < 16 && width < rows) {
    const int next = 2 * width;
    const long long ctas = static_cast<long long>(n_groups) * next;
    if (entries / next < kUnionFewEntries || (next == 16 && ctas > 128)) break;
    if (ctas > sms && entries / width < kUnionManyEntries) break;
    if (at_once(next) < n_groups) break;
    width = next;
  }
  return width;
}

}  // namespace lt
