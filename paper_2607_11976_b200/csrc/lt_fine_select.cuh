// Select-and-sort of one row by one CTA: the kk best of n scored keys, in (score descending, index ascending) order.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "lt_common.cuh"

namespace lt {

// ---------------------------------------------------------------------------------------------
// Distribution sort.  The scores are mapped monotonically to kFineBins bins over their own range, so that a bin of
// the part that matters holds a handful of keys; one histogram and its prefix sum give every bin its place in the
// output, every key up to the bin that holds the kk-th one is dropped into its bin's slots, and a key's final rank
// is its bin's start plus the number of larger keys (full 64-bit keys: score, then index) in the same bin.  Two
// shared-memory atomics and a few comparisons per key and seven barriers per row: latency-bound, which is why the
// keys of a row are held in registers between the sweeps and three CTAs share an SM.  It replaces a least-significant-
// digit radix sort (three to four passes of match.any ranking, ~40 barriers) preceded by a histogram select.  One B200, final
// select of the whole chunk: 4096 rows of 2048 out of 3.4 k candidates 431 -> 137 us, out of 4.2 k 425 -> 153 us, 8192
// rows 736 -> 235 us, one row 23 -> 13 us; 1024 rows with heavy-tailed scores 216 -> 48 us, of tie-ridden ones 187 -> 45 us.
//
// Two mappings are tried: equal-width bins in the score (bell-shaped tails, whole rows around zero), and equal-width bins in
// the score's ordered bit pattern (heavy tails: the width then grows with the score; and rows with NaN scores, which rank by it).  Rows
// that crowd into few bins under both - mass ties above all - are left to the caller: the function then returns false, on every
// thread, without having written anything.
//
// Bound by instructions where many rows are in flight, and by the 40 registers a thread may have with three CTAs to an SM: the range is
// taken in floats, a bin is a difference, an FMA that rounds to a whole number and a clamp, and the first batch's registers are
// given up before the second mapping.  Final select, 4096 rows of 3.4 k candidates 119 -> 94 us, 8192 rows 244 -> 197; first chunk's
// 4096 rows of up to 4096 keys 86 -> 82.  (Bins narrower at the low end, where candidates are densest: 105 us; comparing two or four
// keys of a bin at a time: no better.)
//
//   load(i)   score bits and index of the i-th key, i < n; called several times, for the first batch only where the first mapping fails
//   c         the first kFineBatch * kThreads keys, key j * kThreads + tid in c[j] (anything past n)
//   keys      key_cap 64-bit slots, bins: kFineBins counters (both shared memory)
//   leave_nan rows with a NaN among their scores are left to the caller too
// ---------------------------------------------------------------------------------------------
constexpr int kFineBins = 4096;
constexpr int kFineBatch = 8;

// visits every key of this thread from number `from` on.  kInLoop: the caller goes through several rows.  Registers that only some paths
// set then count as held from one row to the next - those of every sweep together, half a kilobyte a thread went to memory - so
// that the keys past the end are set too.  (Where a CTA selects one row it costs a few instructions: 8 x 16 K dense 13.4 -> 13.6 us.)
template <int kThreads, bool kInLoop, class Load, class Visit>
__device__ __forceinline__ void fine_sweep(const Load& load, unsigned int from, unsigned int n, Visit&& visit) {
  const unsigned int tid = threadIdx.x;
  for (unsigned int at = from; at < n; at += kFineBatch * kThreads) {
    uint2 e[kFineBatch];
#pragma unroll
    for (int j = 0; j < kFineBatch; ++j) {
      if (at + j * kThreads + tid < n) e[j] = load(at + j * kThreads + tid);
      else if (kInLoop) e[j] = make_uint2(0u, 0u);
    }
#pragma unroll
    for (int j = 0; j < kFineBatch; ++j)
      if (at + j * kThreads + tid < n) visit(e[j]);
  }
}

// ... and all of them, the first batch from registers
template <int kThreads, bool kInLoop, class Load, class Visit>
__device__ __forceinline__ void fine_sweep(const Load& load, const uint2 (&c)[kFineBatch], unsigned int n, Visit&& visit) {
  const unsigned int tid = threadIdx.x;
#pragma unroll
  for (int j = 0; j < kFineBatch; ++j)
    if (j * kThreads + tid < n) visit(c[j]);
  fine_sweep<kThreads, kInLoop>(load, kFineBatch * kThreads, n, visit);
}

// One attempt: sweep(visit) visits every key of the thread, bin_of(score bits) maps monotonically, the best keys to bin 0; the bins are
// zero, and a barrier lies behind that.  False, and nothing written, where the keys crowd.
template <int kThreads, class Sweep, class BinOf>
__device__ __forceinline__ bool fine_attempt(const Sweep& sweep, int kk, int topk, uint64_t* keys, unsigned int key_cap,
                                             unsigned int* bins, int32_t* out_idx, float* out_score, int n_keys, Control* ctl,
                                             const BinOf& bin_of) {
  constexpr int kWarps = kThreads / 32;
  constexpr int kBinsPerThread = kFineBins / kThreads;
  static_assert(kWarps <= 32 && kBinsPerThread % 4 == 0, "one warp combines the warps' results; bins are swept in 16-byte pieces");
  __shared__ unsigned int s_sum[kWarps], s_cost[kWarps];
  __shared__ unsigned int s_keep, s_last_bin;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  uint4* bins4 = reinterpret_cast<uint4*>(bins);
  sweep([&](uint2 e) { atomicAdd(&bins[bin_of(e.x)], 1u); });
  __syncthreads();
  // starts of the bins, and the number of comparisons the bins up to the kk-th key will take
  unsigned int cnt[kBinsPerThread], mine = 0;
#pragma unroll
  for (int j = 0; j < kBinsPerThread / 4; ++j) {
    const uint4 v = bins4[tid * (kBinsPerThread / 4) + j];
    cnt[4 * j] = v.x;
    cnt[4 * j + 1] = v.y;
    cnt[4 * j + 2] = v.z;
    cnt[4 * j + 3] = v.w;
    mine += v.x + v.y + v.z + v.w;
  }
  unsigned int incl = mine;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const unsigned int o = __shfl_up_sync(0xffffffffu, incl, d);
    if (lane >= d) incl += o;
  }
  if (lane == 31) s_sum[warp] = incl;
  __syncthreads();
  const unsigned int before = __reduce_add_sync(0xffffffffu, lane < warp ? s_sum[lane] : 0u);
  unsigned int run = before + incl - mine;
  unsigned int cost = 0;
#pragma unroll
  for (int j = 0; j < kBinsPerThread; ++j) {
    const unsigned int m = cnt[j];
    cnt[j] = run;
    if (run < static_cast<unsigned int>(kk)) {
      cost += min(m, 16383u) * min(m, 16383u);  // the sum stays below 2^32 for the largest capacity (12 * LT_MAX_TOPK keys)
      if (run + m >= static_cast<unsigned int>(kk)) {  // exactly one bin
        s_keep = run + m;
        s_last_bin = tid * kBinsPerThread + j;
      }
    }
    run += m;
  }
#pragma unroll
  for (int j = 0; j < kBinsPerThread / 4; ++j)
    bins4[tid * (kBinsPerThread / 4) + j] = make_uint4(cnt[4 * j], cnt[4 * j + 1], cnt[4 * j + 2], cnt[4 * j + 3]);
  cost = __reduce_add_sync(0xffffffffu, cost);
  if (lane == 0) s_cost[warp] = cost;
  __syncthreads();
  const unsigned int keep = s_keep, last_bin = s_last_bin;
  cost = __reduce_add_sync(0xffffffffu, lane < kWarps ? s_cost[lane] : 0u);
  // comparisons past a few dozen per key cost more than the caller's sort
  if (keep > key_cap || cost > 48u * keep + 65536u) {
    __syncthreads();  // everybody has read the verdict before the bins are cleared or the caller reuses them
    return false;
  }
  // every kept key to the next free slot of its bin; bins[b] ends as the end of bin b
  sweep([&](uint2 e) {
    const unsigned int b = bin_of(e.x);
    if (b <= last_bin) keys[atomicAdd(&bins[b], 1u)] = (static_cast<uint64_t>(score_to_key(e.x)) << 32) | (0xffffffffu - e.y);
  });
  __syncthreads();
  for (unsigned int i = tid; i < keep; i += kThreads) {
    const uint64_t key = keys[i];
    const unsigned int b = bin_of(key_to_score_bits(static_cast<unsigned int>(key >> 32)));
    unsigned int rank = b > 0u ? bins[b - 1] : 0u;
    const unsigned int end = bins[b];
    for (unsigned int j = rank; j < end; ++j) rank += keys[j] > key ? 1u : 0u;
    if (rank < static_cast<unsigned int>(kk)) {
      const bool have = LT_IN_BOUNDS(key_index(key) >= 0 && key_index(key) < n_keys, ctl);  // never publish an index outside the keys
      out_idx[rank] = have ? key_index(key) : -1;
      if (out_score != nullptr) out_score[rank] = have ? key_score(key) : -INFINITY;
    }
  }
  for (int j = kk + tid; j < topk; j += kThreads) {
    out_idx[j] = -1;
    if (out_score != nullptr) out_score[j] = -INFINITY;
  }
  return true;
}

template <int kThreads, bool kInLoop = false, class Load>
__device__ __forceinline__ bool fine_select_sort(const Load& load, const uint2 (&c)[kFineBatch], unsigned int n, int kk, int topk,
                                                 uint64_t* keys, unsigned int key_cap, unsigned int* bins, int32_t* out_idx,
                                                 float* out_score, int n_keys, Control* ctl, bool leave_nan = false) {
  constexpr int kWarps = kThreads / 32;
  __shared__ unsigned int s_min[kWarps], s_max[kWarps];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  auto clear_bins = [&]() {
    for (int i = tid; i < kFineBins / 4; i += kThreads) reinterpret_cast<uint4*>(bins)[i] = make_uint4(0u, 0u, 0u, 0u);
  };
  // range of the scores; a warp with a NaN among its own says so in place of its maximum
  float fmin = INFINITY, fmax = -INFINITY;
  bool nan = false;
  fine_sweep<kThreads, kInLoop>(load, c, n, [&](uint2 e) {
    const float v = __uint_as_float(e.x);
    fmin = fminf(fmin, v);
    fmax = fmaxf(fmax, v);
    nan = nan || v != v;
  });
  // (reduced as ordered bit patterns, of which a NaN's is the largest)
  unsigned int kmin = __reduce_min_sync(0xffffffffu, score_to_key(__float_as_uint(fmin)));
  unsigned int kmax = __reduce_max_sync(0xffffffffu, nan ? 0xffffffffu : score_to_key(__float_as_uint(fmax)));
  if (lane == 0) {
    s_min[warp] = kmin;
    s_max[warp] = kmax;
  }
  clear_bins();
  __syncthreads();
  kmin = __reduce_min_sync(0xffffffffu, s_min[lane % kWarps]);
  kmax = __reduce_max_sync(0xffffffffu, s_max[lane % kWarps]);
  nan = kmax == 0xffffffffu;
  if (nan && leave_nan) {
    __syncthreads();
    return false;
  }
  if (!nan) {
    // (the sum with 2^23 rounds to a whole number, the bin, in the low bits; every step rounds monotonically.  Infinite scores give
    // NaNs and infinities: patterns above the last bin's)
    constexpr float kOne = 8388608.f;
    constexpr unsigned int kOneBits = 0x4b000000u;
    fmin = __uint_as_float(key_to_score_bits(kmin));
    fmax = __uint_as_float(key_to_score_bits(kmax));
    const float scale = static_cast<float>(kFineBins) / (fmax - fmin);
    if (fine_attempt<kThreads>([&](auto&& visit) { fine_sweep<kThreads, kInLoop>(load, c, n, visit); }, kk, topk, keys, key_cap, bins, out_idx, out_score, n_keys, ctl, [&](uint32_t bits) {
          const float d = fmax - __uint_as_float(bits);
          const float b = __fmaf_rn(d, scale, kOne);
          return min(__float_as_uint(b), kOneBits + kFineBins - 1u) - kOneBits;
        }))
      return true;
    clear_bins();
  }
  // equal-width bins in the ordered bit patterns.  (Rare: the keys are all loaded again, so that the registers of the first batch are free
  // beyond the first attempt.)
  if (nan) {
    kmin = 0xffffffffu;
    kmax = 0u;
    fine_sweep<kThreads, kInLoop>(load, 0u, n, [&](uint2 e) {
      kmin = min(kmin, score_to_key(e.x));
      kmax = max(kmax, score_to_key(e.x));
    });
    kmin = __reduce_min_sync(0xffffffffu, kmin);
    kmax = __reduce_max_sync(0xffffffffu, kmax);
    __syncthreads();  // the range without NaNs has been read
    if (lane == 0) {
      s_min[warp] = kmin;
      s_max[warp] = kmax;
    }
    __syncthreads();
    kmin = __reduce_min_sync(0xffffffffu, s_min[lane % kWarps]);
    kmax = __reduce_max_sync(0xffffffffu, s_max[lane % kWarps]);
  } else {
    __syncthreads();  // the bins are clear
  }
  const unsigned int span = kmax - kmin;
  const unsigned int kscale = span >= kFineBins ? static_cast<unsigned int>((static_cast<unsigned long long>(kFineBins) << 32) / (static_cast<unsigned long long>(span) + 1ull)) : 0u;
  return fine_attempt<kThreads>([&](auto&& visit) { fine_sweep<kThreads, kInLoop>(load, 0u, n, visit); }, kk, topk, keys, key_cap, bins, out_idx, out_score, n_keys, ctl, [&](uint32_t bits) {
    const unsigned int k = score_to_key(bits);
    return kscale != 0u ? __umulhi(kmax - k, kscale) : min(kmax - k, static_cast<unsigned int>(kFineBins - 1));
  });
}

}  // namespace lt
