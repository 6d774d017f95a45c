// Previous-chunk sampler (paper Sec. 3.2 "Sampling"): count how often each key position occurs in a
// chunk's top-k result, rank the counts, and gather the keys of a caller-provided sample into a dense buffer that the
// scan kernel can score through an ordinary tensor map.  Integer / byte work only.
#include <cuda_runtime.h>
#include <stdint.h>

#include "lt_common.cuh"
#include "lt_host.h"

namespace lt {

namespace {

// counts[p] += 1 for every entry p of idx with 0 <= p < N (fire-and-forget atomics; 16-byte loads)
__global__ void __launch_bounds__(256) count_positions_kernel(const int32_t* __restrict__ idx, long long n, int N,
                                                              unsigned int* __restrict__ counts) {
  chain_wait();
  const long long stride = static_cast<long long>(gridDim.x) * blockDim.x;
  long long i = static_cast<long long>(blockIdx.x) * blockDim.x + threadIdx.x;
  const long long n4 = ((reinterpret_cast<uintptr_t>(idx) & 15u) == 0) ? n / 4 : 0;
  const int4* idx4 = reinterpret_cast<const int4*>(idx);
  for (long long j = i; j < n4; j += stride) {
    const int4 v = __ldg(idx4 + j);
    if (static_cast<unsigned int>(v.x) < static_cast<unsigned int>(N)) atomicAdd(counts + v.x, 1u);
    if (static_cast<unsigned int>(v.y) < static_cast<unsigned int>(N)) atomicAdd(counts + v.y, 1u);
    if (static_cast<unsigned int>(v.z) < static_cast<unsigned int>(N)) atomicAdd(counts + v.z, 1u);
    if (static_cast<unsigned int>(v.w) < static_cast<unsigned int>(N)) atomicAdd(counts + v.w, 1u);
  }
  for (long long j = n4 * 4 + i; j < n; j += stride) {
    const int v = __ldg(idx + j);
    if (static_cast<unsigned int>(v) < static_cast<unsigned int>(N)) atomicAdd(counts + v, 1u);
  }
}

// ---- ranking the counts: top n_out of the N distinct keys (count, position) ---------------------------------------
// A key packs the count above the complemented position, (count << pos_bits) | (2^pos_bits - 1 - position), so that
// larger keys mean (count descending, position ascending) and only count_bits + pos_bits bits carry information.
// A grid-wide MSB radix select, one launch per 11-bit digit of those bits: every CTA histograms the digit of the
// keys that still match the prefix found so far (per-thread run-length aggregation: neighbouring positions mostly
// share the digit), adds its counters to the global histogram, and the last CTA to finish picks the digit in
// which the count from the top reaches the number of keys still wanted.  The keys are distinct (the position is
// part of them), so after the last digit the prefix IS the n_out-th largest key and no tie needs ranking.  A pass over a few MB is a
// chain of latencies (loads, merge, pick), so there are as few passes as shared memory counts cheaply, and the pick is a
// prefix sum by the whole CTA.  Whole call, 1024 x 2048
// entries over 262,144 positions, 6144 wanted, 76 -> 48 us; 512 x 512 over 1,000,003, 1536 wanted, 66 -> 35 (8-bit digits, picked by one
// thread, and two launches for the order).
constexpr int kRankBits = 11;
constexpr int kRankDigits = 1 << kRankBits;
constexpr int kRankThreads = 512;
constexpr int kOrderKeys = 256;  // keys ranked by one CTA
struct RankState {
  unsigned long long prefix;
  unsigned int remaining;
  unsigned int done;
  unsigned int n_written;
  unsigned int slices_done[(LT_MAX_TOPK + kOrderKeys - 1) / kOrderKeys];
};
// Scratch: the state, then the passes' histogram, over which the keys are written once the passes are through, then the keys' ranks.
constexpr size_t kRankStateBytes = 1280;
constexpr size_t kRankHistBytes = kRankDigits * 4;
static_assert(sizeof(RankState) <= kRankStateBytes, "state block");
__host__ __device__ inline unsigned int* rank_hist(RankState* st) { return reinterpret_cast<unsigned int*>(reinterpret_cast<uint8_t*>(st) + kRankStateBytes); }
size_t rank_keys_bytes(int n_out) { return static_cast<size_t>(n_out) * 8 > kRankHistBytes ? static_cast<size_t>(n_out) * 8 : kRankHistBytes; }

constexpr int kRankBatch = 8;  // loads a thread keeps in flight (one CTA-wide load per batch entry)

__device__ __forceinline__ unsigned long long rank_key(unsigned int count, unsigned int pos, int pos_bits) {
  return (static_cast<unsigned long long>(count) << pos_bits) | ((1ull << pos_bits) - 1ull - pos);
}
// inclusive prefix sum over the CTA (kRankThreads threads); the barrier inside separates what precedes it from what follows
__device__ __forceinline__ unsigned int cta_inclusive_sum(unsigned int v, unsigned int* warp_sum) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  unsigned int incl = v;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const unsigned int o = __shfl_up_sync(0xffffffffu, incl, d);
    if (lane >= d) incl += o;
  }
  if (lane == 31) warp_sum[warp] = incl;
  __syncthreads();
  return incl + __reduce_add_sync(0xffffffffu, lane < warp ? warp_sum[lane] : 0u);
}

__global__ void __launch_bounds__(kRankThreads) rank_pass_kernel(const unsigned int* __restrict__ counts, int N, RankState* st, int shift,
                                                                 int first_pass, int pos_bits, int want) {
  __shared__ __align__(16) unsigned int hist[kRankDigits];
  __shared__ unsigned int warp_sum[kRankThreads / 32];
  __shared__ bool last;
  constexpr int kPer = kRankDigits / kRankThreads;
  static_assert(kPer == 4, "a thread's digits are one 16-byte piece");
  const int tid = threadIdx.x;
  const unsigned long long mask = first_pass ? 0ull : (~0ull << (shift + kRankBits));
  unsigned int* const total = rank_hist(st);
  reinterpret_cast<uint4*>(hist)[tid] = make_uint4(0u, 0u, 0u, 0u);
  chain_wait();
  const unsigned long long prefix = st->prefix;
  __syncthreads();
  unsigned int run_digit = kRankDigits, run_len = 0;
  // each CTA walks one contiguous range of positions with coalesced loads, kRankBatch of them in flight per
  // thread (one load at a time is latency-bound: 16 dependent DRAM round trips per pass); a thread's consecutive
  // keys are a CTA's width apart, which still share their leading digits (the count's high bits)
  const int per_thread = (N + gridDim.x * blockDim.x - 1) / (gridDim.x * blockDim.x);
  const long long first = static_cast<long long>(blockIdx.x) * blockDim.x * per_thread + threadIdx.x;
  for (int j0 = 0; j0 < per_thread; j0 += kRankBatch) {
    unsigned int c[kRankBatch];
#pragma unroll
    for (int u = 0; u < kRankBatch; ++u) {
      const long long i = first + static_cast<long long>(j0 + u) * blockDim.x;
      c[u] = (j0 + u < per_thread && i < N) ? __ldg(counts + i) : 0u;
    }
#pragma unroll
    for (int u = 0; u < kRankBatch; ++u) {
      const long long i = first + static_cast<long long>(j0 + u) * blockDim.x;
      if (j0 + u >= per_thread || i >= N) continue;
      const unsigned long long key = rank_key(c[u], static_cast<unsigned int>(i), pos_bits);
      if ((key & mask) != prefix) continue;
      const unsigned int digit = static_cast<unsigned int>(key >> shift) & (kRankDigits - 1u);
      if (digit == run_digit) {
        ++run_len;
      } else {
        if (run_len > 0) atomicAdd(&hist[run_digit], run_len);
        run_digit = digit;
        run_len = 1;
      }
    }
  }
  if (run_len > 0) atomicAdd(&hist[run_digit], run_len);
  __syncthreads();
#pragma unroll
  for (int j = 0; j < kPer; ++j) {
    const unsigned int n = hist[tid + j * kRankThreads];
    if (n != 0u) atomicAdd(total + tid + j * kRankThreads, n);
  }
  __threadfence();
  __syncthreads();
  if (tid == 0) last = atomicAdd(&st->done, 1u) == gridDim.x - 1;
  __syncthreads();
  if (!last) return;
  __threadfence();
  // digits from the top down, four per thread: the one in which the count reaches what is still wanted
  const int low = kRankDigits - kPer * (tid + 1);  // this thread's lowest digit
  const uint4 h = __ldcg(reinterpret_cast<const uint4*>(total + low));
  const unsigned int remaining = first_pass ? static_cast<unsigned int>(want) : st->remaining;
  const unsigned int mine = h.x + h.y + h.z + h.w;
  const unsigned int incl = cta_inclusive_sum(mine, warp_sum);
  unsigned int cum = incl - mine;
  if (cum < remaining && incl >= remaining) {  // exactly one thread: there are N >= want keys
    const unsigned int c[kPer] = {h.w, h.z, h.y, h.x};
    int digit = -1;
#pragma unroll
    for (int j = 0; j < kPer; ++j) {
      if (digit < 0 && cum + c[j] >= remaining) digit = low + kPer - 1 - j;
      if (digit < 0) cum += c[j];
    }
    st->remaining = remaining - cum;
    st->prefix = prefix | (static_cast<unsigned long long>(digit) << shift);
    st->done = 0;
  }
  *reinterpret_cast<uint4*>(total + low) = make_uint4(0u, 0u, 0u, 0u);
}

// every key at or above the n_out-th largest goes to the list (any order; exactly n_out of them): places are reserved once for each CTA
// and round of kRankBatch keys per thread (a reservation per warp and key, all on one address, took twice as long)
__global__ void __launch_bounds__(kRankThreads) rank_collect_kernel(const unsigned int* __restrict__ counts, int N, RankState* st,
                                                                    unsigned long long* __restrict__ keys, int n_out, int pos_bits) {
  __shared__ unsigned int warp_sum[kRankThreads / 32];
  __shared__ unsigned int s_base;
  chain_wait();
  const unsigned long long kth = st->prefix;
  const int per_thread = (N + gridDim.x * blockDim.x - 1) / (gridDim.x * blockDim.x);
  const long long first = static_cast<long long>(blockIdx.x) * blockDim.x * per_thread + threadIdx.x;
  for (int j0 = 0; j0 < per_thread; j0 += kRankBatch) {
    unsigned int c[kRankBatch];
#pragma unroll
    for (int u = 0; u < kRankBatch; ++u) {
      const long long i = first + static_cast<long long>(j0 + u) * blockDim.x;
      c[u] = (j0 + u < per_thread && i < N) ? __ldg(counts + i) : 0u;
    }
    unsigned int take = 0;
#pragma unroll
    for (int u = 0; u < kRankBatch; ++u) {
      const long long i = first + static_cast<long long>(j0 + u) * blockDim.x;
      if (j0 + u < per_thread && i < N && rank_key(c[u], static_cast<unsigned int>(i), pos_bits) >= kth) take |= 1u << u;
    }
    const unsigned int mine = __popc(take);
    const unsigned int incl = cta_inclusive_sum(mine, warp_sum);
    if (threadIdx.x == kRankThreads - 1) s_base = incl != 0u ? atomicAdd(&st->n_written, incl) : 0u;
    __syncthreads();
    unsigned int pos = s_base + incl - mine;
#pragma unroll
    for (int u = 0; u < kRankBatch; ++u) {
      const long long i = first + static_cast<long long>(j0 + u) * blockDim.x;
      if ((take >> u) & 1u) {
        if (pos < static_cast<unsigned int>(n_out)) keys[pos] = rank_key(c[u], static_cast<unsigned int>(i), pos_bits);
        ++pos;
      }
    }
    __syncthreads();  // the sums have been read
  }
}

// Order of the n_out winners (count descending, position ascending) by counting: the keys are distinct, so the
// number of larger keys IS a key's place in the output.  CTA (x, y) ranks kOrderKeys keys against slice y of the list
// held in shared memory; the slices' partial ranks meet in `rank` (zeroed by the caller), and the last CTA of a block of keys writes them
// out.  n_out^2 comparisons spread over the whole GPU take a few microseconds where a one-CTA sort of the list took 80; slices of 256 keys
// fill it from a few thousand keys on.
constexpr int kOrderSlice = 256;

__global__ void __launch_bounds__(kOrderKeys) rank_order_kernel(const unsigned long long* __restrict__ keys, int n_out, RankState* st,
                                                                unsigned int* __restrict__ rank, int pos_bits, int32_t* __restrict__ out_pos,
                                                                int32_t* __restrict__ out_count) {
  __shared__ __align__(16) unsigned long long slice[kOrderSlice];
  __shared__ bool last;
  static_assert(kOrderSlice == kOrderKeys, "a thread fetches one key of the slice");
  chain_wait();
  const int me = blockIdx.x * kOrderKeys + threadIdx.x, other = blockIdx.y * kOrderSlice + threadIdx.x;
  const unsigned long long mine = me < n_out ? keys[me] : ~0ull;
  slice[threadIdx.x] = other < n_out ? keys[other] : 0ull;  // (zero is larger than nothing)
  __syncthreads();
  unsigned int larger = 0;
#pragma unroll 16
  for (int i = 0; i < kOrderSlice; i += 2) {
    const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(slice + i);
    larger += (v.x > mine ? 1u : 0u) + (v.y > mine ? 1u : 0u);
  }
  if (larger != 0u) atomicAdd(rank + me, larger);
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) last = atomicAdd(&st->slices_done[blockIdx.x], 1u) == gridDim.y - 1;
  __syncthreads();
  if (!last || me >= n_out) return;
  __threadfence();
  const unsigned int r = __ldcg(rank + me);
  if (r >= static_cast<unsigned int>(n_out)) return;  // cannot happen for distinct keys
  out_pos[r] = static_cast<int32_t>((1ull << pos_bits) - 1ull - (mine & ((1ull << pos_bits) - 1ull)));
  if (out_count != nullptr) out_count[r] = static_cast<int32_t>(mine >> pos_bits);
}

// out_k[j] = key row at position sample_idx[j] (or j * stride when no list is given), row_bytes bytes (a
// multiple of 16); out_scale[j] = its scale.  One 16-byte piece per thread; positions outside [0, N) are read as
// position 0.  With a paged key cache the position is translated to its physical row first.
__global__ void __launch_bounds__(256) gather_keys_kernel(const uint8_t* __restrict__ k, const float* __restrict__ k_scale,
                                                          const int32_t* __restrict__ sample_idx, long long stride,
                                                          int n_sample, int N, int row_bytes,
                                                          const int* __restrict__ page_table, long long pool_rows,
                                                          Control* ctl, uint8_t* __restrict__ out_k,
                                                          float* __restrict__ out_scale) {
  chain_wait();
  const int pieces = row_bytes >> 4;
  const long long g = static_cast<long long>(blockIdx.x) * blockDim.x + threadIdx.x;
  const long long j = g / pieces;
  const int piece = static_cast<int>(g - j * pieces);
  if (j >= n_sample) return;
  long long s = sample_idx != nullptr ? static_cast<long long>(__ldg(sample_idx + j)) : j * stride;
  if (s < 0 || s >= N) s = 0;
  if (page_table != nullptr) {
    s = static_cast<long long>(__ldg(page_table + s / kPageKeys)) * kPageKeys + s % kPageKeys;
    if (!LT_IN_BOUNDS(s >= 0 && s < pool_rows, ctl)) s = 0;  // a page-table entry outside the pool
  }
  const uint4 v = __ldg(reinterpret_cast<const uint4*>(k + static_cast<size_t>(s) * row_bytes) + piece);
  reinterpret_cast<uint4*>(out_k + static_cast<size_t>(j) * row_bytes)[piece] = v;
  if (piece == 0 && k_scale != nullptr) out_scale[j] = __ldg(k_scale + s);
}

}  // namespace

cudaError_t launch_count_positions(const int32_t* idx, long long n, int N, unsigned int* counts, cudaStream_t stream) {
  if (n <= 0) return cudaSuccess;
  long long blocks = (n / 4 + 255) / 256;
  if (blocks < 1) blocks = 1;
  if (blocks > 16 * sm_count()) blocks = 16 * sm_count();
  return launch_chained(count_positions_kernel, static_cast<unsigned int>(blocks), 256, 0, stream, 1, idx, n, N, counts);
}

// (for LT_MAX_TOPK keys, which every workspace is sized for, what it was with a smaller histogram inside the state)
size_t rank_scratch_bytes(int n_out) { return kRankStateBytes + rank_keys_bytes(n_out) + static_cast<size_t>(n_out) * 4; }

namespace {
int bits_for(unsigned long long max_value) {
  int b = 1;
  while (b < 64 && (max_value >> b) != 0ull) ++b;
  return b;
}
}  // namespace

// Ranks the N counts and writes the n_out most frequent positions; scratch: rank_scratch_bytes(n_out) bytes, zeroed,
// 256-byte aligned.  max_count: an upper bound of any count (it fixes how many digits the select has to visit).
cudaError_t launch_rank_counts(const unsigned int* counts, int N, int n_out, unsigned long long max_count, void* scratch,
                               int32_t* out_pos, int32_t* out_count, cudaStream_t stream) {
  RankState* st = static_cast<RankState*>(scratch);
  unsigned long long* keys = reinterpret_cast<unsigned long long*>(rank_hist(st));
  unsigned int* rank = reinterpret_cast<unsigned int*>(reinterpret_cast<uint8_t*>(keys) + rank_keys_bytes(n_out));
  if (max_count > 0xffffffffull) max_count = 0xffffffffull;
  const int pos_bits = bits_for(static_cast<unsigned long long>(N - 1));
  const int passes = (bits_for(max_count) + pos_bits + kRankBits - 1) / kRankBits;
  int blocks = (N + kRankThreads * kRankBatch - 1) / (kRankThreads * kRankBatch);
  if (blocks < 1) blocks = 1;
  if (blocks > 2 * sm_count()) blocks = 2 * sm_count();
  cudaError_t e = cudaSuccess;
  for (int pass = 0; pass < passes && e == cudaSuccess; ++pass)
    e = launch_chained(rank_pass_kernel, blocks, kRankThreads, 0, stream, 1, counts, N, st, kRankBits * (passes - 1 - pass), pass == 0 ? 1 : 0, pos_bits, n_out);
  if (e == cudaSuccess) e = launch_chained(rank_collect_kernel, blocks, kRankThreads, 0, stream, 1, counts, N, st, keys, n_out, pos_bits);
  if (e == cudaSuccess)
    e = launch_chained(rank_order_kernel, dim3((n_out + kOrderKeys - 1) / kOrderKeys, (n_out + kOrderSlice - 1) / kOrderSlice), kOrderKeys, 0, stream, 1,
                       keys, n_out, st, rank, pos_bits, out_pos, out_count);
  return e;
}

cudaError_t launch_gather_keys(const void* k, const float* k_scale, const int32_t* sample_idx, long long stride, int n_sample,
                               int N, int row_bytes, const int* page_table, long long pool_rows, Control* ctl, void* out_k,
                               float* out_scale, cudaStream_t stream) {
  const long long threads = static_cast<long long>(n_sample) * (row_bytes >> 4);
  return launch_chained(gather_keys_kernel, static_cast<unsigned int>((threads + 255) / 256), 256, 0, stream, 1,
                        static_cast<const uint8_t*>(k), k_scale, sample_idx, stride, n_sample, N, row_bytes, page_table, pool_rows, ctl,
                        static_cast<uint8_t*>(out_k), out_scale);
}

}  // namespace lt
