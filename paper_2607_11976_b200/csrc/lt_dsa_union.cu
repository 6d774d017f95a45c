// LiteDSA union list + membership masks (paper Sec. 3.3): a cluster of CTAs per group of adjacent query rows marks the
// group's selected key positions in a bit-packed bitmap in shared memory (atomic OR, so a position selected by several
// rows is kept once), sweeps the bitmap into one ascending list shared by the group, and gives every row a bitmask
// over the list's slots.  Integer work only.
//
// Bound by the outputs: every list slot and every mask word is written once, ones, zeros and padding alike, with
// coalesced stores, and the index matrix is read twice (the second time from L2).  Each CTA of a cluster owns a few of
// the group's rows: it marks them in its own copy of the bitmap, the copies are combined word by word through
// distributed shared memory (a CTA combines one slice and hands it to all), and from then on every CTA can turn a
// position into its slot on its own: it writes its slice of the list and builds its rows' masks in shared memory.
// With one CTA per group, outputs cleared by memsets and masks built by global atomics, 4096 rows x 2048 over 128 K
// positions in groups of 64 took 201 us; now 46 us, with 25 us the time of
// moving the bytes.  What is left is the chain of phases of a CTA (mark 5 us, combine 5, prefix 2, list 4, then the masks) and
// clusters that fill some GPCs' SMs with four CTAs and others' with three.
#include <cooperative_groups.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "lt_cluster_width.h"
#include "lt_common.cuh"
#include "lt_host.h"

namespace lt {

namespace {

// Bitmap words per pass, words to a stored prefix and words of the mask buffer.  The longer the context, the more of the shared
// memory the bitmap takes: up to 262,144 positions a prefix per word, up to 1,048,576 (128 KB of bitmap) one per 4 words, beyond
// that windows of 1,572,864 positions (192 KB) with one per 8 - or of 1,048,576, where a mask does not fit the smaller buffer
// beside the large window (each piece of a mask looks all entries up again).
constexpr int kWordPrefixMax = 8192;
constexpr int kFourPrefixMax = 32768;
constexpr int kWindowWords = 49152;
constexpr int kMaskBufWords = 4096;      // 131,072 slots
constexpr int kMaskBufWordsWide = 2048;  // ... beside a bitmap of 192 KB
constexpr int kUnionWideEntries = 2048;  // see the launch

struct UnionParams {
  const int32_t* idx;   // [T][topk]
  int T, topk, N, group;
  int rows_per_cta;
  int cap;              // group * topk: slots of one group's list
  int mask_words;       // ceil(cap / 32)
  int window_words;     // bitmap words kept at once (a multiple of 8)
  int buf_words;        // words of the mask buffer (a multiple of 4)
  int32_t* union_pos;   // [n_groups][cap]
  int32_t* union_len;   // [n_groups]
  uint32_t* mask;       // [T][mask_words]
};

// (a multiple of four: the masks behind the prefix are accessed in 16-byte pieces)
__host__ __device__ constexpr int prefix_words(int unit, int window_words) { return unit == 1 ? window_words : (window_words / unit + 3) / 4 * 4; }

__device__ __forceinline__ unsigned int popc4(uint4 v) { return __popc(v.x) + __popc(v.y) + __popc(v.z) + __popc(v.w); }

__device__ __forceinline__ unsigned int warp_inclusive_sum(unsigned int v, int lane) {
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const unsigned int o = __shfl_up_sync(0xffffffffu, v, d);
    if (lane >= d) v += o;
  }
  return v;
}

// the slot of position q of the window, whose first slot is `slot`
template <int kUnit>
__device__ __forceinline__ unsigned int slot_of(const uint32_t* bitmap, const uint32_t* prefix, unsigned int q, unsigned int slot) {
  const uint4* bitmap4 = reinterpret_cast<const uint4*>(bitmap);
  const unsigned int below = (1u << (q & 31)) - 1u;
  if (kUnit == 1) {
    slot += prefix[q >> 5] + __popc(bitmap[q >> 5] & below);
  } else {
    const uint4 v = bitmap4[q >> 7];
    const unsigned int k = (q >> 5) & 3u;
    const uint32_t word = k == 0u ? v.x : k == 1u ? v.y : k == 2u ? v.z : v.w;
    if (kUnit == 8 && ((q >> 7) & 1u) != 0u) slot += popc4(bitmap4[(q >> 7) - 1u]);
    slot += prefix[(q >> 5) / kUnit] + __popc(word & below) + (k > 0u ? __popc(v.x) : 0) + (k > 1u ? __popc(v.y) : 0) + (k > 2u ? __popc(v.z) : 0);
  }
  return slot;
}

// kUnit: words to a stored prefix (1, 4 or 8).  512 threads while several CTAs share an SM, 1024 where one has it to itself.
// kWholeRows: one window, and rows whose masks come one at a time and whole, four positions to a thread, in 16-byte pieces.  Kernels of
// their own: beside that loop the general one was slower (4096 x 2048 in 32 groups over 65,536 positions 76.2 -> 78.3 us).
// Where four CTAs share an SM a thread has 32 registers, and it counts what holds them: copies of the masks are not unrolled (the same 73.3, in 64
// groups, whole rows, 41.9 -> 40.1).
template <int kUnit, int kUnionThreads, bool kWholeRows>
__global__ void __launch_bounds__(kUnionThreads, kUnionThreads == 1024 ? 1 : kUnit == 1 ? 4 : 2) dsa_union_kernel(const UnionParams p) {
  constexpr int kUnionWarps = kUnionThreads / 32;
  namespace cg = cooperative_groups;
  cg::cluster_group cl = cg::this_cluster();
  const int n_cta = static_cast<int>(cl.num_blocks()), rank = static_cast<int>(cl.block_rank());
  extern __shared__ __align__(16) uint32_t smem_u[];
  uint32_t* bitmap = smem_u;
  uint32_t* prefix = bitmap + p.window_words;  // list slots before every kUnit words (within the window)
  uint32_t* masks = prefix + prefix_words(kUnit, p.window_words);
  __shared__ unsigned int warp_tot[kUnionWarps];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int grp = static_cast<int>(blockIdx.x) / n_cta;
  const int r1 = min(p.T, (grp + 1) * p.group);
  const int row_lo = min(r1, grp * p.group + rank * p.rows_per_cta), row_hi = min(r1, row_lo + p.rows_per_cta);
  const int32_t* my_idx = p.idx + static_cast<size_t>(row_lo) * p.topk;
  const int n_entries = (row_hi - row_lo) * p.topk;  // at most group * topk <= 2^24
  int32_t* out = p.union_pos + static_cast<size_t>(grp) * p.cap;
  unsigned int list_len = 0;  // entries of earlier windows (uniform across the cluster)

  for (int i = tid; i < p.buf_words; i += kUnionThreads) masks[i] = 0u;
  chain_wait();
  for (long long wbase = 0; kWholeRows || wbase < p.N; wbase += static_cast<long long>(p.window_words) * 32) {
    const long long left = p.N - wbase;
    const int span = kWholeRows ? p.N : static_cast<int>(left < static_cast<long long>(p.window_words) * 32 ? left : static_cast<long long>(p.window_words) * 32);
    const bool last = left <= static_cast<long long>(p.window_words) * 32;
    const int words = ((span + 31) / 32 + 7) / 8 * 8;
    const int base = kWholeRows ? 0 : static_cast<int>(wbase);  // positions are below N < 2^31
    for (int i = tid; i < words / 4; i += kUnionThreads) reinterpret_cast<uint4*>(bitmap)[i] = make_uint4(0u, 0u, 0u, 0u);
    __syncthreads();
    // 1. mark this CTA's rows: the atomic OR deduplicates
    auto mark = [&](int pos) {
      const unsigned int q = static_cast<unsigned int>(pos - base);
      if (pos >= base && q < static_cast<unsigned int>(span)) atomicOr(&bitmap[q >> 5], 1u << (q & 31));
    };
    int done = 0;
    if ((reinterpret_cast<uintptr_t>(my_idx) & 15u) == 0) {
      const int4* v4 = reinterpret_cast<const int4*>(my_idx);
      const int n4 = n_entries / 4;
      for (int i = tid; i < n4; i += 4 * kUnionThreads) {
        int4 v[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) v[j] = __ldg(v4 + min(i + j * kUnionThreads, n4 - 1));  // marking an entry twice is harmless
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          mark(v[j].x);
          mark(v[j].y);
          mark(v[j].z);
          mark(v[j].w);
        }
      }
      done = n4 * 4;
    }
    for (int i = done + tid; i < n_entries; i += kUnionThreads) mark(__ldg(my_idx + i));
    cl.sync();
    // 2. combine: this CTA ORs one slice of all copies and writes it back to all of them
    const int slice = ((words + n_cta - 1) / n_cta + 7) / 8 * 8;
    const int s0 = min(words, rank * slice), s1 = min(words, s0 + slice);
    if (n_cta > 1) {
      for (int i = s0 / 4 + tid; i < s1 / 4; i += kUnionThreads) {
        uint4 v = make_uint4(0u, 0u, 0u, 0u);
#pragma unroll 8
        for (int r = 0; r < n_cta; ++r) {
          const uint4 o = reinterpret_cast<const uint4*>(cl.map_shared_rank(bitmap, r))[i];
          v.x |= o.x;
          v.y |= o.y;
          v.z |= o.z;
          v.w |= o.w;
        }
#pragma unroll 8
        for (int r = 0; r < n_cta; ++r) reinterpret_cast<uint4*>(cl.map_shared_rank(bitmap, r))[i] = v;
      }
      cl.sync();
    }
    // 3. list slots before every unit: each warp owns a run of consecutive groups of 32 pieces of 4 (or 8) words, a piece per lane
    const uint4* bitmap4 = reinterpret_cast<const uint4*>(bitmap);
    const int units = words / (kUnit == 8 ? 8 : 4);
    auto popc_piece = [&](int u) { return kUnit == 8 ? popc4(bitmap4[2 * u]) + popc4(bitmap4[2 * u + 1]) : popc4(bitmap4[u]); };
    const int groups = (units + 31) / 32;
    const int per_warp = (groups + kUnionWarps - 1) / kUnionWarps;
    const int u0 = min(groups, warp * per_warp) * 32, u1 = min(units, u0 + per_warp * 32);
    unsigned int mine = 0;
    for (int u = u0 + lane; u < u1; u += 32) mine += popc_piece(u);
    mine = __reduce_add_sync(0xffffffffu, mine);
    if (lane == 0) warp_tot[warp] = mine;
    __syncthreads();
    const unsigned int wt = lane < kUnionWarps ? warp_tot[lane] : 0u;
    const unsigned int total = __reduce_add_sync(0xffffffffu, wt);
    unsigned int run = __reduce_add_sync(0xffffffffu, lane < warp ? wt : 0u);
    for (int u = u0; u < u1; u += 32) {
      const unsigned int c = u + lane < u1 ? popc_piece(u + lane) : 0u;
      const unsigned int incl = warp_inclusive_sum(c, lane);
      if (u + lane < u1) {
        const unsigned int before = run + incl - c;
        if (kUnit == 1) {
          const uint4 v = bitmap4[u + lane];
          const unsigned int p1 = before + __popc(v.x), p2 = p1 + __popc(v.y), p3 = p2 + __popc(v.z);
          reinterpret_cast<uint4*>(prefix)[u + lane] = make_uint4(before, p1, p2, p3);
        } else {
          prefix[u + lane] = before;
        }
      }
      run += __shfl_sync(0xffffffffu, incl, 31);
    }
    __syncthreads();
    // 4. sweep: the set bits of this CTA's slice to consecutive slots.  32 words at a time: well-filled ones a word per
    // warp and step, which coalesces the stores, sparse ones (a context much longer than the list) a word per lane
    for (int w = s0 + warp * 32; w < s1; w += kUnionThreads) {
      const uint32_t own = w + lane < s1 ? bitmap[w + lane] : 0u;
      const unsigned int in_all = __reduce_add_sync(0xffffffffu, static_cast<unsigned int>(__popc(own)));
      if (in_all == 0u) continue;
      int32_t* dst = kWholeRows ? out : out + list_len;
      if (in_all >= 96u) {
        dst += prefix[w / kUnit];  // (w is a multiple of eight)
#pragma unroll 8
        for (int j = 0; j < 32; ++j) {
          const uint32_t word = __shfl_sync(0xffffffffu, own, j);
          if ((word >> lane) & 1u) dst[__popc(word & ((1u << lane) - 1u))] = base + (w + j) * 32 + lane;
          dst += __popc(word);
        }
      } else if (kUnit == 8) {  // (a scan over the warp is shorter than the set bits of up to seven words of the unit)
        const unsigned int c = __popc(own);
        dst += prefix[w / kUnit] + warp_inclusive_sum(c, lane) - c;
        for (uint32_t word = own; word != 0u; word &= word - 1u) *dst++ = base + (w + lane) * 32 + __ffs(word) - 1;
      } else if (own != 0u) {
        dst += prefix[(w + lane) / kUnit];
        if (kUnit == 4) {
          const uint4 v = bitmap4[(w + lane) >> 2];
          const int k = lane & 3;
          dst += (k > 0 ? __popc(v.x) : 0) + (k > 1 ? __popc(v.y) : 0) + (k > 2 ? __popc(v.z) : 0);
        }
        for (uint32_t word = own; word != 0u; word &= word - 1u) *dst++ = base + (w + lane) * 32 + __ffs(word) - 1;
      }
    }
    // 5. membership: slot of a position = slots before its unit + set bits before it inside the unit.  Masks are built in
    // shared memory and written out whole: as many rows at a time as a buffer takes, or buf_words words of one row.  The
    // word in which this window's slots begin also holds bits of the window before, which the same CTA wrote.
    const int w_first = static_cast<int>(list_len >> 5);
    const unsigned int end_slot = list_len + total;
    const int w_end = last ? p.mask_words : static_cast<int>((end_slot + 31u) >> 5);
    const int batch = p.mask_words <= p.buf_words ? p.buf_words / p.mask_words : 1;
    if constexpr (kWholeRows) {
      // a row's positions are fetched while the mask of the row before it is written out (4096 x 2048 in 64 groups over 131,072 positions
      // 63.0 -> 46.0 us)
      const bool mine = 4 * tid < p.topk;
      const int4* src = reinterpret_cast<const int4*>(my_idx) + tid;
      uint4* dst = reinterpret_cast<uint4*>(p.mask + static_cast<size_t>(row_lo) * p.mask_words);
      uint4* masks4 = reinterpret_cast<uint4*>(masks);
      auto member = [&](int pos) {
        if (static_cast<unsigned int>(pos) < static_cast<unsigned int>(span)) {
          const unsigned int slot = slot_of<kUnit>(bitmap, prefix, static_cast<unsigned int>(pos), 0u);
          atomicOr(&masks[slot >> 5], 1u << (slot & 31));
        }
      };
      int4 next = make_int4(-1, -1, -1, -1);
      if (mine && row_lo < row_hi) next = __ldg(src);
      for (int left_rows = row_hi - row_lo; left_rows > 0; --left_rows) {
        const int4 pos = next;
        src += p.topk / 4;
        if (mine && left_rows > 1) next = __ldg(src);
        member(pos.x);
        member(pos.y);
        member(pos.z);
        member(pos.w);
        __syncthreads();
        // written and cleared by the same thread
#pragma unroll 1
        for (int i = tid; i < p.mask_words / 4; i += kUnionThreads) {
          dst[i] = masks4[i];
          masks4[i] = make_uint4(0u, 0u, 0u, 0u);
        }
        dst += p.mask_words / 4;
        __syncthreads();
      }
      list_len = total;
      break;
    } else {
      for (int w0 = w_first; w0 < w_end; w0 += p.buf_words) {
        const int n_words = min(w_end - w0, p.buf_words);
        const bool has_bits = (static_cast<unsigned int>(w0) << 5) < end_slot;
        for (int row = row_lo; row < row_hi; row += batch) {
          uint32_t* buf = masks;
          const int rows = min(batch, row_hi - row);
          __syncthreads();  // the batch before has been written out
          if (has_bits) {
            const int32_t* e = p.idx + static_cast<size_t>(row) * p.topk;
            const int n = rows * p.topk;
            for (int i = tid; i < n; i += 4 * kUnionThreads) {
              int pos[4];
#pragma unroll
              for (int j = 0; j < 4; ++j) pos[j] = __ldg(e + min(i + j * kUnionThreads, n - 1));  // (the last entry again: harmless)
#pragma unroll
              for (int j = 0; j < 4; ++j) {
                const unsigned int q = static_cast<unsigned int>(pos[j] - base);
                if (pos[j] < base || q >= static_cast<unsigned int>(span)) continue;
                const unsigned int slot = slot_of<kUnit>(bitmap, prefix, q, list_len);
                const int mw = static_cast<int>(slot >> 5) - w0;
                const int r = rows == 1 ? 0 : min(i + j * kUnionThreads, n - 1) / p.topk;
                if (mw >= 0 && mw < n_words) atomicOr(&buf[r * n_words + mw], 1u << (slot & 31));
              }
            }
            if (w0 == w_first && (list_len & 31u) != 0u && tid < rows)
              atomicOr(&buf[tid * n_words], __ldcg(p.mask + static_cast<size_t>(row + tid) * p.mask_words + w0));
          }
          __syncthreads();
          // written and cleared by the same thread
          uint32_t* dst = p.mask + static_cast<size_t>(row) * p.mask_words + w0;
          if (rows == 1 || n_words == p.mask_words) {  // one run of words
            const int n = rows * n_words;
            if ((reinterpret_cast<uintptr_t>(dst) & 15u) == 0 && (n & 3) == 0) {
#pragma unroll 1
              for (int i = tid; i < n / 4; i += kUnionThreads) {
                reinterpret_cast<uint4*>(dst)[i] = reinterpret_cast<const uint4*>(buf)[i];
                reinterpret_cast<uint4*>(buf)[i] = make_uint4(0u, 0u, 0u, 0u);
              }
            } else {
              for (int i = tid; i < n; i += kUnionThreads) {
                dst[i] = buf[i];
                buf[i] = 0u;
              }
            }
          } else {
            for (int r = 0; r < rows; ++r)
              for (int i = tid; i < n_words; i += kUnionThreads) {
                dst[static_cast<size_t>(r) * p.mask_words + i] = buf[r * n_words + i];
                buf[r * n_words + i] = 0u;
              }
          }
        }
      }
      list_len = end_slot;
      __syncthreads();
    }
  }
  for (unsigned int i = list_len + static_cast<unsigned int>(rank * kUnionThreads + tid); i < static_cast<unsigned int>(p.cap);
       i += static_cast<unsigned int>(n_cta * kUnionThreads))
    out[i] = -1;
  if (rank == 0 && tid == 0) p.union_len[grp] = static_cast<int32_t>(list_len);
}

}  // namespace

cudaError_t launch_dsa_union(const int32_t* idx, int T, int topk, int N, int group, int32_t* union_pos, int32_t* union_len,
                             uint32_t* mask, cudaStream_t stream) {
  UnionParams p{};
  p.idx = idx;
  p.T = T;
  p.topk = topk;
  p.N = N;
  p.group = group;
  p.cap = group * topk;
  p.mask_words = (p.cap + 31) / 32;
  p.union_pos = union_pos;
  p.union_len = union_len;
  p.mask = mask;
  const int n_groups = (T + group - 1) / group;
  const int words = (static_cast<int>((static_cast<long long>(N) + 31) / 32) + 7) / 8 * 8;
  const int unit = words <= kWordPrefixMax ? 1 : words <= kFourPrefixMax || p.mask_words > kMaskBufWordsWide ? 4 : 8;
  const int window_max = unit == 8 ? kWindowWords : kFourPrefixMax;
  p.window_words = words < window_max ? words : window_max;
  const int buf_max = unit == 8 ? kMaskBufWordsWide : kMaskBufWords;
  const int rows = group < T ? group : T;
  // shared memory with a mask buffer for n rows, or for as much of them as buf_max
  auto shared_bytes = [&](int n) {
    const long long n_words = static_cast<long long>(p.mask_words) * n;
    p.buf_words = n_words < buf_max ? static_cast<int>(n_words + 3) / 4 * 4 : buf_max;
    return (p.window_words + prefix_words(unit, p.window_words) + p.buf_words) * 4;
  };

  // by unit and threads
  static std::atomic<unsigned long long> done[2][5];
  using Kernel = void (*)(UnionParams);
  const Kernel kernels[2][5] = {{dsa_union_kernel<1, 512, false>, dsa_union_kernel<1, 1024, false>, dsa_union_kernel<4, 512, false>,
                                 dsa_union_kernel<4, 1024, false>, dsa_union_kernel<8, 1024, false>},
                                {dsa_union_kernel<1, 512, true>, dsa_union_kernel<1, 1024, true>, dsa_union_kernel<4, 512, true>,
                                 dsa_union_kernel<4, 1024, true>, dsa_union_kernel<8, 1024, true>}};
  const int first = unit == 1 ? 0 : unit == 4 ? 2 : 4;
  cudaError_t e = allow_smem(reinterpret_cast<const void*>(kernels[0][first]), done[0][first], true);
  if (e != cudaSuccess) return e;
  // how many clusters of a width run at once: asked for once for each device, unit, CTAs of that size to an SM, and width (with the
  // largest mask buffer, of one CTA for all rows)
  const int smem_max = shared_bytes(rows);
  const int per_sm = (228 * 1024) / (smem_max + 2048) < 4 ? (228 * 1024) / (smem_max + 2048) : 4;
  static std::atomic<short> at_once_cache[64][3][4][5];
  int dev = 0, sms = 0;
  e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  auto at_once = [&](int width) {
    // (sharing an SM pays CTAs of at most 32 KB of bitmap: 1024 x 2048 over 524,288 positions in 32 groups, width 4 / 8, 31 / 34 us)
    if (unit != 1 && static_cast<long long>(n_groups) * width > sms) return 0;
    int log2 = 0;
    while ((1 << log2) < width) ++log2;
    std::atomic<short>& known = at_once_cache[dev & 63][first / 2][per_sm > 0 ? per_sm - 1 : 0][log2];
    int n = known.load(std::memory_order_relaxed);
    if (n == 0) {
      n = 1 + clusters_at_once(kernels[0][first], unit == 8 ? 1024 : 512, smem_max, width);
      known.store(static_cast<short>(n), std::memory_order_relaxed);
    }
    return n - 1;
  };
  const int width = union_cluster_width(n_groups, rows, static_cast<long long>(rows) * topk, sms, at_once);
  p.rows_per_cta = (rows + width - 1) / width;
  const int smem = shared_bytes(p.rows_per_cta);
  // A CTA with an SM to itself and little to mark is bound by its sweeps over the bitmap: 1024 threads halve them (8 rows x 2048 over
  // 200,000 positions, width 8, 13.6 -> 12.2 us; but 64 x 2048 over 131,072, width 16, 8192 entries a CTA, 17.2 -> 21.1).
  // Wide CTAs do not share an SM, which leaves few places for clusters of 8 (500 x 512 in 16 groups, width 8, 17.4 -> 22.7).  Beside
  // a window of 192 KB there is one CTA to an SM in any case.
  const bool wide = unit == 8 ||
                    (static_cast<long long>(n_groups) * width <= (width == 1 ? sms : unit == 1 ? sms / 2 : 0) &&
                     static_cast<long long>(p.rows_per_cta) * topk <= kUnionWideEntries);
  const int threads = wide ? 1024 : 512;
  // (what the loop over whole rows takes.  Rows that come several at a time wait for their positions at each batch; prefetching them was not tried)
  const bool whole = words <= p.window_words && p.mask_words <= p.buf_words && p.buf_words / p.mask_words == 1 && topk % 4 == 0 && topk <= 4 * threads &&
                     p.mask_words % 4 == 0 && ((reinterpret_cast<uintptr_t>(idx) | reinterpret_cast<uintptr_t>(mask)) & 15u) == 0;
  const int k = unit == 8 || !wide ? first : first + 1;
  e = allow_smem(reinterpret_cast<const void*>(kernels[whole][k]), done[whole][k], true);
  if (e != cudaSuccess) return e;
  return launch_chained(kernels[whole][k], n_groups * width, threads, smem, stream, width, p);
}

}  // namespace lt
