// Shared device helpers for the indexer top-k kernels (sm_100a only).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "../../include/lt_indexer.h"

namespace lt {

constexpr int kBins = LT_BINS;
constexpr int kTileKeys = 128;  // keys per MMA tile (UMMA M)

// ---------------------------------------------------------------------------------------------
// workspace control block (device memory).  One per call.
// ---------------------------------------------------------------------------------------------
struct Control {
  int status;         // LT_STATUS_* bits
  int fb_rows;        // rows that took the fallback
  int max_survivors;  // largest tail[] of any row
  int tot_survivors;  // sum of tail[] (saturating)
  int overflow_rows;  // rows whose candidate buffer overflowed
  int fb_blocks;      // number of entries in the fallback block list
  int pad[2];
};

// The status block opens without a launch of its own: the call's first scan clears it and leaves each CTA's status bits in a byte of its
// own behind it, and the kernel after that, a byte per thread of its first CTA, adds them to the status word.  (A kernel that only
// cleared the block and the counters cost a 1-row call 0.9 of 22.9 us, a first chunk of 4096 rows 2 of 184.)  With more CTAs than bytes,
// everything is cleared ahead of the call.  The bounds-checking build, whose checks write the status word from every kernel, clears the
// block, and nothing else, ahead of the call, and then goes the same way.
constexpr int kStatusSlots = 256 - static_cast<int>(sizeof(Control));  // what the block leaves of its 256 bytes
#if defined(LT_DEBUG_BOUNDS)
constexpr bool kControlClearedAhead = true;
#else
constexpr bool kControlClearedAhead = false;
#endif
__device__ __forceinline__ void clear_control(Control* ctl, int tid) {
  if (!kControlClearedAhead && tid < static_cast<int>(sizeof(Control) / 4)) reinterpret_cast<int*>(ctl)[tid] = 0;
}
// ---------------------------------------------------------------------------------------------
// Index checks of the bounds-checking build (compiled with -DLT_DEBUG_BOUNDS; it stands in for a memory
// checker): LT_IN_BOUNDS(cond, ctl) is `cond`, and where it is false it records LT_STATUS_BOUNDS in the
// status word so that the caller can skip the access and carry on - nothing traps.  In the release build
// it is the constant true and costs nothing.
// ---------------------------------------------------------------------------------------------
#if defined(LT_DEBUG_BOUNDS)
__device__ __forceinline__ bool lt_in_bounds(bool cond, Control* ctl) {
  if (!cond && ctl != nullptr) atomicOr(&ctl->status, LT_STATUS_BOUNDS);
  return cond;
}
#define LT_IN_BOUNDS(cond, ctl) (::lt::lt_in_bounds((cond), (ctl)))
#else
#define LT_IN_BOUNDS(cond, ctl) (true)
#endif

// A scan's CTA leaves its status bits; the kernel behind it fetches them beside its first loads, and looks at them with those.
__device__ __forceinline__ void store_status_slot(unsigned char* slots, Control* ctl, int bits) {
  if (LT_IN_BOUNDS(static_cast<int>(blockIdx.x) < kStatusSlots, ctl)) slots[blockIdx.x] = static_cast<unsigned char>(bits);
}
__device__ __forceinline__ int load_status_slot(const unsigned char* slots, int n_slots, int tid, Control* ctl) {
  return slots != nullptr && blockIdx.x == 0 && tid < n_slots && LT_IN_BOUNDS(n_slots <= kStatusSlots, ctl) ? slots[tid] : 0;
}
__device__ __forceinline__ void add_status(Control* ctl, int slot) {
  if (slot != 0) atomicOr(&ctl->status, slot);
}

// ---------------------------------------------------------------------------------------------
// Chained launches.  Every kernel of a call is launched so that it may start when the kernel ahead of it in the stream has no
// CTA left to end (launch_chained in lt_host.h): its launch latency and set-up then run beside the other's completion and
// memory flush.  chain_wait() returns once everything ahead in the stream has completed and its writes are visible.
// EVERY thread of every kernel launched that way that touches global memory calls chain_wait() before it does, on every
// path: a grid that ended without waiting would let the kernel behind it run ahead of the kernel before it.
// Only the scans of the exact fallback let their successor start earlier than that (chain_trigger): nearly always they have nothing to do,
// and neither has the select behind them (4 rows over 2^20 keys 67.5 -> 64.9 us, 1 row 48.0 -> 45.3).  At the top of every kernel the
// trigger slowed what ran beside the waiting grid, 4096 rows over 2^20 keys 40.0 -> 42.5 ms, 4 rows 73 -> 80 us, 77 rows over 300 K keys
// 238 -> 248 us.  A kernel triggers behind its own chain_wait(), so that what its successor waits for is all that is ahead of it.
// ---------------------------------------------------------------------------------------------
__device__ __forceinline__ void chain_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
// Lets the next kernel of the stream start already.
__device__ __forceinline__ void chain_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// ---------------------------------------------------------------------------------------------
// total order on (score, index): larger key = better.  Scores are canonicalised (-0 -> +0)
// where they are produced, so bit order equals value order.
// ---------------------------------------------------------------------------------------------
__host__ __device__ __forceinline__ uint32_t score_to_key(uint32_t bits) {
  return (bits & 0x80000000u) ? ~bits : (bits | 0x80000000u);
}
__host__ __device__ __forceinline__ uint32_t key_to_score_bits(uint32_t key) {
  return (key & 0x80000000u) ? (key & 0x7fffffffu) : ~key;
}
__device__ __forceinline__ uint64_t pack_key(float score, int idx) {
  return (static_cast<uint64_t>(score_to_key(__float_as_uint(score))) << 32) | (0xffffffffu - static_cast<uint32_t>(idx));
}
__device__ __forceinline__ int key_index(uint64_t key) { return static_cast<int>(0xffffffffu - static_cast<uint32_t>(key)); }
__device__ __forceinline__ float key_score(uint64_t key) {
  return __uint_as_float(key_to_score_bits(static_cast<uint32_t>(key >> 32)));
}

// ---------------------------------------------------------------------------------------------
// Equal-width bins over [s_min, s_max] (paper Sec. 3.2 "Sampling").  Bins are DEFINED by their
// lower edges E(b) = fma(b, width, s_min), b = 1..m-1, evaluated by this one function everywhere:
//   bin(s) = largest b in [1, m-1] with E(b) <= s, or 0 if s < E(1).
// Bin 0 therefore also holds everything below the sampled range, bin m-1 everything above it,
// and "s >= E(b)" is exactly "bin(s) >= b" for b >= 1, which makes the float gate and the
// integer histogram agree bit for bit.  Threshold bin 0 means "accept all".
// ---------------------------------------------------------------------------------------------
__device__ __forceinline__ float bin_edge(int b, float smin, float width) {
  return b <= 0 ? -INFINITY : __fmaf_rn(static_cast<float>(b), width, smin);
}
// `inv_width` is only used for a first guess (1 / width, any rounding); the edge comparisons that
// follow decide, so the result does not depend on it.
__device__ __forceinline__ int bin_of(float s, float smin, float width, float inv_width) {
  if (!(s >= bin_edge(1, smin, width))) return 0;
  if (!(width > 0.f)) return kBins - 1;  // degenerate range: every edge equals s_min
  float g = (s - smin) * inv_width;
  int b = g >= static_cast<float>(kBins - 1) ? kBins - 1 : (g < 1.f ? 1 : static_cast<int>(g));
  while (b < kBins - 1 && s >= bin_edge(b + 1, smin, width)) ++b;
  while (b > 1 && s < bin_edge(b, smin, width)) --b;
  return b;
}
// The bins of two scores side by side: the guesses are right but for scores within rounding of an edge, and only those take bin_of.
__device__ __forceinline__ void bins_of2(float s0, float s1, float smin, float width, float inv_width, int& b0, int& b1) {
  auto guess = [&](float s) {
    const float g = fminf(fmaxf((s - smin) * inv_width, 0.f), static_cast<float>(kBins - 1));
    return static_cast<int>(g);
  };
  // (bin 0 has no lower edge, the last bin no upper one; a zero width leaves every score but those below s_min outside its guess)
  auto off = [&](float s, int b) {
    const float f = static_cast<float>(b);
    return (b > 0 && s < __fmaf_rn(f, width, smin)) || (b < kBins - 1 && s >= __fmaf_rn(f + 1.f, width, smin));
  };
  b0 = guess(s0);
  b1 = guess(s1);
  const bool off0 = off(s0, b0), off1 = off(s1, b1);
  if (off0) b0 = bin_of(s0, smin, width, inv_width);
  if (off1) b1 = bin_of(s1, smin, width, inv_width);
}
__device__ __forceinline__ int bin_of(float s, float smin, float width) {
  return bin_of(s, smin, width, width > 0.f ? 1.f / width : 0.f);
}

// ---------------------------------------------------------------------------------------------
// bitonic sort of n (power of two, >= 2) 64-bit keys in shared memory, descending.  Every thread
// handles whole compare-exchange pairs: pair t of a stage with distance j is (i, i | j) where i is t
// with a zero bit inserted at bit log2(j), so no thread idles on the upper element of a pair.
// ---------------------------------------------------------------------------------------------
__device__ __forceinline__ void bitonic_sort_desc(uint64_t* s, int n, int tid, int nthreads) {
  const int half = n >> 1;
  for (int k = 2; k <= n; k <<= 1) {
    for (int j = k >> 1; j > 0; j >>= 1) {
      for (int t = tid; t < half; t += nthreads) {
        const int i = ((t & ~(j - 1)) << 1) | (t & (j - 1));
        const int ixj = i | j;
        const uint64_t a = s[i], b = s[ixj];
        const bool desc = (i & k) == 0;
        if (desc ? (a < b) : (a > b)) {
          s[i] = b;
          s[ixj] = a;
        }
      }
      __syncthreads();
    }
  }
}

__host__ __device__ __forceinline__ int next_pow2(int v) {
  int p = 1;
  while (p < v) p <<= 1;
  return p;
}

// keys visible to row t
__host__ __device__ __forceinline__ int visible_keys(int t, int N, int causal_offset) {
  long long v = static_cast<long long>(causal_offset) + t + 1;
  return v < 0 ? 0 : (v > N ? N : static_cast<int>(v));
}

}  // namespace lt
