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
// positions in groups of 64 took 201 us; now 69 us, with 25 us the time of
// moving the bytes.  What is left is the chain of phases of a CTA (mark 5 us, combine 5, prefix 2, list 4, masks 20 - 28) and
// clusters that fill some GPCs' SMs with four CTAs and others' with three.
#include <cooperative_groups.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "lt_common.cuh"
#include "lt_host.h"

namespace lt {

namespace {

constexpr int kUnionThreads = 512;
constexpr int kUnionWarps = kUnionThreads / 32;
constexpr int kWindowWords = 32768;     // bitmap words per pass: 1,048,576 positions, 128 KB
constexpr int kWordPrefixMax = 8192;    // windows of up to this many words keep a prefix per word, larger ones per 4 words
constexpr int kMaskBufWords = 4096;     // mask buffer: 131,072 slots

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
__host__ __device__ constexpr int prefix_words(bool per_word, int window_words) { return per_word ? window_words : (window_words / 4 + 3) / 4 * 4; }

__device__ __forceinline__ unsigned int popc4(uint4 v) { return __popc(v.x) + __popc(v.y) + __popc(v.z) + __popc(v.w); }

__device__ __forceinline__ unsigned int warp_inclusive_sum(unsigned int v, int lane) {
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const unsigned int o = __shfl_up_sync(0xffffffffu, v, d);
    if (lane >= d) v += o;
  }
  return v;
}

// kWordPrefix: the window is small enough for a prefix per word
template <bool kWordPrefix>
__global__ void __launch_bounds__(kUnionThreads, kWordPrefix ? 4 : 1) dsa_union_kernel(const UnionParams p) {
  namespace cg = cooperative_groups;
  cg::cluster_group cl = cg::this_cluster();
  const int n_cta = static_cast<int>(cl.num_blocks()), rank = static_cast<int>(cl.block_rank());
  extern __shared__ __align__(16) uint32_t smem_u[];
  uint32_t* bitmap = smem_u;
  uint32_t* prefix = bitmap + p.window_words;  // list slots before every word, or every 4 words (within the window)
  uint32_t* masks = prefix + prefix_words(kWordPrefix, p.window_words);
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
  for (long long wbase = 0; wbase < p.N; wbase += static_cast<long long>(p.window_words) * 32) {
    const long long left = p.N - wbase;
    const int span = static_cast<int>(left < static_cast<long long>(p.window_words) * 32 ? left : static_cast<long long>(p.window_words) * 32);
    const bool last = left <= static_cast<long long>(p.window_words) * 32;
    const int words = ((span + 31) / 32 + 7) / 8 * 8;
    const int base = static_cast<int>(wbase);  // positions are below N < 2^31
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
    // 3. list slots before every 4 words: each warp owns a run of consecutive 128-word groups, 4 words per lane
    const uint4* bitmap4 = reinterpret_cast<const uint4*>(bitmap);
    const int units = words / 4;
    const int groups = (units + 31) / 32;
    const int per_warp = (groups + kUnionWarps - 1) / kUnionWarps;
    const int u0 = min(groups, warp * per_warp) * 32, u1 = min(units, u0 + per_warp * 32);
    unsigned int mine = 0;
    for (int u = u0 + lane; u < u1; u += 32) mine += popc4(bitmap4[u]);
    mine = __reduce_add_sync(0xffffffffu, mine);
    if (lane == 0) warp_tot[warp] = mine;
    __syncthreads();
    const unsigned int wt = lane < kUnionWarps ? warp_tot[lane] : 0u;
    const unsigned int total = __reduce_add_sync(0xffffffffu, wt);
    unsigned int run = __reduce_add_sync(0xffffffffu, lane < warp ? wt : 0u);
    for (int u = u0; u < u1; u += 32) {
      const unsigned int c = u + lane < u1 ? popc4(bitmap4[u + lane]) : 0u;
      const unsigned int incl = warp_inclusive_sum(c, lane);
      if (u + lane < u1) {
        const unsigned int before = run + incl - c;
        if (kWordPrefix) {
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
      const unsigned int c = __popc(own);
      const unsigned int incl = warp_inclusive_sum(c, lane);
      int32_t* dst = out + list_len + prefix[kWordPrefix ? w : w >> 2];
      if (__shfl_sync(0xffffffffu, incl, 31) >= 96u) {
#pragma unroll 8
        for (int j = 0; j < 32; ++j) {
          const uint32_t word = __shfl_sync(0xffffffffu, own, j);
          if ((word >> lane) & 1u) dst[__popc(word & ((1u << lane) - 1u))] = base + (w + j) * 32 + lane;
          dst += __popc(word);
        }
      } else {
        dst += incl - c;
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
              const unsigned int below = (1u << (q & 31)) - 1u;
              unsigned int slot = list_len;
              if (kWordPrefix) {
                slot += prefix[q >> 5] + __popc(bitmap[q >> 5] & below);
              } else {
                const uint4 v = bitmap4[q >> 7];
                const unsigned int k = (q >> 5) & 3u;
                const uint32_t word = k == 0u ? v.x : k == 1u ? v.y : k == 2u ? v.z : v.w;
                slot += prefix[q >> 7] + __popc(word & below) + (k > 0u ? __popc(v.x) : 0) + (k > 1u ? __popc(v.y) : 0) + (k > 2u ? __popc(v.z) : 0);
              }
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
  p.window_words = words < kWindowWords ? words : kWindowWords;
  const bool word_prefix = p.window_words <= kWordPrefixMax;
  // As many CTAs per group as it has rows and as run at the same time: a CTA that waits for a second wave pays the clearing,
  // combining and sweeping of its copy of the bitmap all over (4096 x 2048 over 1 M positions in 64 groups: width 2 / 4 / 8
  // 106 / 117 / 188 us; over 128 K positions 103 / 72 / 69 us).  Sixteen CTAs need a whole GPC: only for few groups.
  const int resident = 148 * (word_prefix ? 4 : 1);
  int width = 1;
  while (width < 8 && width < group && n_groups * width * 2 <= resident) width <<= 1;
  if (width == 8 && group >= 16 && n_groups * 16 <= 128) width = 16;
  p.rows_per_cta = (group + width - 1) / width;
  // the buffer holds all of a CTA's rows, or as much as kMaskBufWords
  const long long all_rows = static_cast<long long>(p.mask_words) * p.rows_per_cta;
  p.buf_words = all_rows < kMaskBufWords ? static_cast<int>(all_rows + 3) / 4 * 4 : kMaskBufWords;
  const int smem = (p.window_words + prefix_words(word_prefix, p.window_words) + p.buf_words) * 4;
  static std::atomic<unsigned long long> done[2];
  auto kernel = word_prefix ? dsa_union_kernel<true> : dsa_union_kernel<false>;
  cudaError_t e = allow_smem(reinterpret_cast<const void*>(kernel), done[word_prefix ? 1 : 0], true);
  if (e != cudaSuccess) return e;
  return launch_chained(kernel, n_groups * width, kUnionThreads, smem, stream, width, p);
}

}  // namespace lt
