// Selection-side kernels of the indexer top-k: sample statistics, final select over the candidate
// buffers, full-row radix select (generic path, unfused baseline, exact fallback) and the generic
// SIMT scoring kernel.
#include <cooperative_groups.h>
#include <cuda_bf16.h>
#include <cuda_fp8.h>
#include <cuda_runtime.h>
#include <float.h>
#include <math.h>
#include <stdint.h>

#include "lt_cluster_width.h"
#include "lt_common.cuh"
#include "lt_fine_select.cuh"
#include "lt_host.h"

namespace lt {

namespace {

constexpr int kSelBatch = 8;  // independent row loads in flight per thread of the full-row select
constexpr int kSelCap = 2 * LT_MAX_TOPK;  // 64-bit keys the final select can sort in shared memory

// ---------------------------------------------------------------------------------------------
// generic SIMT scoring (any H, D, dtype).  Bound by fp32 FMA issue once there is enough of it: a thread keeps 4 keys x 8
// heads of dots in registers (three 16-byte shared loads per 32 FMAs), a warp covers 128 keys of one query row, the eight
// warps of a CTA share the key tile (kRows query rows x 8 / kRows runs of 128 keys).  With a thread per key that fetched
// both operands of every FMA, 64 x 4096 x 8 heads x 64 took 49 us and
// 128 x 16384 x 32 x 128 2659 us; now 14 and 457 us (half of the fp32 FMA peak).  Warps without a row only help to stage: with their
// FMAs 1 x 20001 x 32 x 128, nine CTAs more than SMs, took 65 us, now 36 for the scores.  Dots run over d and the head sum over h in
// ascending order, one FMA each: every launch shape gives the same bits.
// ---------------------------------------------------------------------------------------------
template <int kDtype>
__device__ __forceinline__ float load_elem(const void* base, size_t i) {
  if (kDtype == LT_DTYPE_F32) return reinterpret_cast<const float*>(base)[i];
  if (kDtype == LT_DTYPE_BF16) return __uint_as_float(static_cast<uint32_t>(reinterpret_cast<const uint16_t*>(base)[i]) << 16);
  __half_raw hr = __nv_cvt_fp8_to_halfraw(reinterpret_cast<const uint8_t*>(base)[i], __NV_E4M3);
  return __half2float(__half(hr));
}

__global__ void __launch_bounds__(256) zero_kernel(uint4* p, long long n) {
  chain_wait();
  for (long long i = static_cast<long long>(blockIdx.x) * 256 + threadIdx.x; i < n; i += static_cast<long long>(gridDim.x) * 256)
    p[i] = make_uint4(0u, 0u, 0u, 0u);
}

constexpr int kSimtThreads = 256;
constexpr int kSimtD = 16;           // coordinates staged at a time
constexpr int kSimtHeads = 8;        // heads in registers
constexpr int kSimtKeyPad = 4;       // (keeps 16-byte alignment, spreads the transposing stores over the banks)

template <int kDtype, int kRows>
__global__ void __launch_bounds__(kSimtThreads, 2) simt_scores_kernel(const void* __restrict__ q, const float* __restrict__ w,
                                                                   const void* __restrict__ k, const float* __restrict__ k_scale, int N,
                                                                   int H, int D, int causal_offset, int row_begin, int row_end,
                                                                   float* __restrict__ out, long long ld, Control* clear_ctl) {
  constexpr int kKeys = 128 * (8 / kRows);  // keys of the CTA's tile
  __shared__ __align__(16) float ks[kSimtD][kKeys + kSimtKeyPad];
  __shared__ __align__(16) float qs[kRows][kSimtD][kSimtHeads];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int t0 = row_begin + blockIdx.y * kRows, s0 = blockIdx.x * kKeys;
  const int tr = warp % kRows, t = t0 + tr;
  const int key = (warp / kRows) * 128 + lane * 4;  // first of the thread's four keys in the tile
  // the next piece of both operands travels in registers while the current one is worked on
  constexpr int kK = kKeys * kSimtD / kSimtThreads, kQ = kRows * kSimtHeads * kSimtD / kSimtThreads;
  static_assert(kK * kSimtThreads == kKeys * kSimtD && kQ * kSimtThreads == kRows * kSimtHeads * kSimtD, "whole loads per thread");
  float kr[kK], qr[kQ];
  // thread -> (coordinate d, key sj + 16 j) and (coordinate d, head hj, row rj + 2 j)
  static_assert(kSimtThreads == 256 && kSimtD == 16 && kSimtHeads == 8, "the index arithmetic below");
  const int dj = tid & 15, sj = tid >> 4, hj = (tid >> 4) & 7, rj = tid >> 7;
  const size_t k_at = static_cast<size_t>(s0 + sj) * D + dj, q_at = (static_cast<size_t>(t0 + rj) * H + hj) * D + dj;
  const int live = min(kK, (N - s0 - sj + 15) / 16);  // keys of this thread that exist (may be negative)
  auto fetch = [&](int h0, int d0) {
    const bool in = d0 + dj < D;
#pragma unroll
    for (int j = 0; j < kK; ++j) kr[j] = in && j < live ? load_elem<kDtype>(k, k_at + d0 + static_cast<size_t>(j) * 16 * D) : 0.f;
#pragma unroll
    for (int j = 0; j < kQ; ++j)
      qr[j] = in && h0 + hj < H && t0 + rj + 2 * j < row_end
                  ? load_elem<kDtype>(q, q_at + static_cast<size_t>(h0) * D + d0 + static_cast<size_t>(j) * 2 * H * D) : 0.f;
  };
  chain_wait();
  // the status block of the call, which only later kernels write to
  if (clear_ctl != nullptr && blockIdx.x == 0 && blockIdx.y == 0 && tid < static_cast<int>(sizeof(Control) / 4)) reinterpret_cast<int*>(clear_ctl)[tid] = 0;
  fetch(0, 0);
  float total[4] = {0.f, 0.f, 0.f, 0.f};
  for (int h0 = 0; h0 < H; h0 += kSimtHeads) {
    float acc[kSimtHeads][4];
#pragma unroll
    for (int h = 0; h < kSimtHeads; ++h)
#pragma unroll
      for (int j = 0; j < 4; ++j) acc[h][j] = 0.f;
    for (int d0 = 0; d0 < D; d0 += kSimtD) {
      __syncthreads();
#pragma unroll
      for (int j = 0; j < kK; ++j) ks[dj][sj + 16 * j] = kr[j];
#pragma unroll
      for (int j = 0; j < kQ; ++j) qs[rj + 2 * j][dj][hj] = qr[j];
      __syncthreads();
      if (d0 + kSimtD < D) {
        fetch(h0, d0 + kSimtD);
      } else if (h0 + kSimtHeads < H) {
        fetch(h0 + kSimtHeads, 0);
      }
      if (t >= row_end) continue;  // a warp without a row leaves the FMA units to the others
#pragma unroll
      for (int d = 0; d < kSimtD; ++d) {
        const float4 kv = *reinterpret_cast<const float4*>(&ks[d][key]);
        const float4 qa = *reinterpret_cast<const float4*>(&qs[tr][d][0]), qb = *reinterpret_cast<const float4*>(&qs[tr][d][4]);
        const float qv[kSimtHeads] = {qa.x, qa.y, qa.z, qa.w, qb.x, qb.y, qb.z, qb.w};
#pragma unroll
        for (int h = 0; h < kSimtHeads; ++h) {
          acc[h][0] = __fmaf_rn(qv[h], kv.x, acc[h][0]);
          acc[h][1] = __fmaf_rn(qv[h], kv.y, acc[h][1]);
          acc[h][2] = __fmaf_rn(qv[h], kv.z, acc[h][2]);
          acc[h][3] = __fmaf_rn(qv[h], kv.w, acc[h][3]);
        }
      }
    }
    if (t < row_end) {
#pragma unroll
      for (int h = 0; h < kSimtHeads; ++h) {
        const float wh = h0 + h < H ? __ldg(w + static_cast<size_t>(t) * H + h0 + h) : 0.f;
#pragma unroll
        for (int j = 0; j < 4; ++j) total[j] = __fmaf_rn(wh, fmaxf(acc[h][j], 0.f), total[j]);
      }
    }
  }
  if (t >= row_end) return;
  const int vis = visible_keys(t, N, causal_offset);
  float* dst = out + static_cast<size_t>(t - row_begin) * ld + s0 + key;
  float v[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const int s = s0 + key + j;
    if (k_scale != nullptr && s < N) total[j] *= k_scale[s];
    v[j] = s < vis ? total[j] + 0.f : -INFINITY;  // -0 -> +0
  }
  if (s0 + key + 3 < N && (reinterpret_cast<uintptr_t>(dst) & 15u) == 0) {
    *reinterpret_cast<float4*>(dst) = make_float4(v[0], v[1], v[2], v[3]);
  } else {
#pragma unroll
    for (int j = 0; j < 4; ++j)
      if (s0 + key + j < N) dst[j] = v[j];
  }
}

// ---------------------------------------------------------------------------------------------
// sample statistics: one CTA per row.  With the default rank, a twentieth of the sample or less, the threshold is nearly always in the upper
// bins: a row's scores stay in registers between the sweep for the range and the one for the histogram (longer rows are
// read again), and only scores from bin kStatsCutBin up are looked at; they are compacted per warp, because a bin search is long and nearly
// every 32 scores hold one.  Rows whose rank-th score lies below the cut - a few outliers stretch their range - count the others too.
// One B200, 8192 rows of 4064 scores 91 -> 54 us, 4096 of 2048 30 -> 25, 1024 of 6144 22 -> 19, against a bin search for every score;
// 4096 of 2048 with outliers 27 -> 35.
// Where the rank is topk - a caller's sample of usually 3 topk positions, sample_rank = -1 - nearly every row would take both sweeps, and a
// short sample is counted before it is sorted out: all scores are counted at once there, and read again for it.  Cut / all, us: 4096
// rows of 6144, rank 2048, 90 / 62; 2048 of 12288, rank 2048 79 / 62, 1024 60 / 62, 512 54 / 62; of 2048, rank 256 19 / 17; 8192 of 1024, rank
// 109, 44 / 35, of 1664 44 / 42, of 2048 46 / 48.
// ---------------------------------------------------------------------------------------------
constexpr int kStatsCutBin = 160;    // of kBins: for bell-shaped scores about a fifth of them, three times the usual rank
constexpr int kStatsHighShare = 8;   // the cut is used for ranks below an eighth of the sample
constexpr int kStatsShort = 2048;    // ... of at least so many scores
template <int kThreads, int kKeep>  // kKeep: scores a thread holds; 0: all scores are counted at once
__global__ void __launch_bounds__(kThreads) sample_stats_kernel(const float* __restrict__ sample, int n_sample, int rank,
                                                                float* __restrict__ smin_out, float* __restrict__ width_out,
                                                                float* __restrict__ thr_out, const OpenParams open) {
  constexpr int kWarps = kThreads / 32;
  __shared__ float red_min[kWarps], red_max[kWarps];
  __shared__ __align__(16) unsigned int hist[kBins];
  __shared__ float high[kWarps][(kKeep > 0 ? kKeep : 1) * 32];  // per warp: its scores from the cut up
  __shared__ int s_more;
  const int t = blockIdx.x;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const float* row = sample + static_cast<size_t>(t) * n_sample;
  chain_wait();
  const int slot = load_status_slot(open.status_slots, open.n_slots, tid, open.ctl);
  if (open.ctl != nullptr) {
    for (int i = tid; i < kBins; i += kThreads) open.hist[static_cast<size_t>(t) * kBins + i] = 0u;
    if (tid == 0) {
      open.tail[t] = 0u;
      open.row_flag[t] = 0;
      const int block = t / open.rows_per_block;
      if (t == block * open.rows_per_block && LT_IN_BOUNDS(block < open.n_blocks, open.ctl)) open.block_flag[block] = 0u;
    }
    if (open.n_slots == 0 && t == 0) clear_control(open.ctl, tid);
  }
  // NaN scores (sums that overflowed) would leave the row without bins; neither the minimum nor the maximum takes them, they
  // are in no bin above 0, and the gate lets none pass
  const float kNan = __uint_as_float(0x7fffffffu);
  float v[kKeep > 0 ? kKeep : 1];
#pragma unroll
  for (int j = 0; j < kKeep; ++j) v[j] = tid + j * kThreads < n_sample ? row[tid + j * kThreads] : kNan;
  add_status(open.ctl, slot);
  float mn = INFINITY, mx = -INFINITY;
#pragma unroll
  for (int j = 0; j < kKeep; ++j) {
    mn = fminf(mn, v[j]);
    mx = fmaxf(mx, v[j]);
  }
  if (kKeep == 0) {
    for (int base = tid; base < n_sample; base += 8 * kThreads) {
      float x[8];
#pragma unroll
      for (int j = 0; j < 8; ++j) x[j] = base + j * kThreads < n_sample ? row[base + j * kThreads] : kNan;
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        mn = fminf(mn, x[j]);
        mx = fmaxf(mx, x[j]);
      }
    }
  } else {
#pragma unroll 8
    for (int i = tid + kKeep * kThreads; i < n_sample; i += kThreads) {
      const float x = row[i];
      mn = fminf(mn, x);
      mx = fmaxf(mx, x);
    }
  }
  auto warp_range = [&]() {
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) {
      mn = fminf(mn, __shfl_xor_sync(0xffffffffu, mn, d));
      mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, d));
    }
  };
  warp_range();
  if (lane == 0) {
    red_min[warp] = mn;
    red_max[warp] = mx;
  }
  for (int i = tid; i < kBins; i += kThreads) hist[i] = 0u;
  __syncthreads();
  mn = red_min[lane % kWarps];
  mx = red_max[lane % kWarps];
  warp_range();
  const float smin = n_sample > 0 ? mn : 0.f;
  const float width = n_sample > 0 ? (mx - smin) / static_cast<float>(kBins) : 0.f;
  const float inv_width = width > 0.f ? 1.f / width : 0.f;
  const float cut = bin_edge(kKeep > 0 ? kStatsCutBin : 0, smin, width);
  auto count = [&](float x) { atomicAdd(&hist[bin_of(x, smin, width, inv_width)], 1u); };
  int n_high = 0;
#pragma unroll
  for (int j = 0; j < kKeep; ++j) {
    const bool take = v[j] >= cut;
    const unsigned int ballot = __ballot_sync(0xffffffffu, take);
    if (take) high[warp][n_high + __popc(ballot & ((1u << lane) - 1u))] = v[j];
    n_high += __popc(ballot);
  }
  __syncwarp();
#pragma unroll 1
  for (int i = lane; i < n_high; i += 32) count(high[warp][i]);
#pragma unroll 2
  for (int i = tid + kKeep * kThreads; i < n_sample; i += kThreads) {
    const float x = row[i];
    if (x >= cut) count(x);
  }
  __syncthreads();
  for (int sweep = 0;; ++sweep) {
    if (warp == 0) {
      // threshold bin = bin holding the rank-th largest sampled score; 0 (accept all) if the sample is smaller than that
      const uint4 h0 = reinterpret_cast<const uint4*>(hist)[lane * 2], h1 = reinterpret_cast<const uint4*>(hist)[lane * 2 + 1];
      const unsigned int c[8] = {h0.x, h0.y, h0.z, h0.w, h1.x, h1.y, h1.z, h1.w};
      const unsigned int mine = c[0] + c[1] + c[2] + c[3] + c[4] + c[5] + c[6] + c[7];
      unsigned int incl = mine;
#pragma unroll
      for (int d = 1; d < 32; d <<= 1) {
        const unsigned int o = __shfl_down_sync(0xffffffffu, incl, d);
        if (lane + d < 32) incl += o;
      }
      const unsigned int need = static_cast<unsigned int>(rank);
      unsigned int cum = incl - mine;
      const bool here = cum < need && incl >= need;
      int tb = 0;
      if (here) {
#pragma unroll
        for (int j = 7; j >= 0; --j) {
          cum += c[j];
          if (tb == 0 && cum >= need) tb = lane * 8 + j;
        }
      }
      const bool found = __any_sync(0xffffffffu, here);
      tb = __reduce_max_sync(0xffffffffu, tb);
      if (lane == 0) {
        s_more = !found && sweep == 0 ? 1 : 0;
        smin_out[t] = smin;
        width_out[t] = width;
        thr_out[t] = bin_edge(tb, smin, width);
      }
    }
    __syncthreads();
    if (s_more == 0) return;
    // the others
#pragma unroll 2
    for (int i = tid; i < n_sample; i += kThreads) {
      const float x = row[i];
      if (!(x >= cut)) count(x);
    }
    __syncthreads();
  }
}

// ---------------------------------------------------------------------------------------------
// Bitonic sort of the first `count` keys of sel[] (shared, room for next_pow2(count)), then the row's outputs.  For rows
// the distribution sort gives up on.
// ---------------------------------------------------------------------------------------------
__device__ __forceinline__ void sort_and_write(uint64_t* sel, int count, int topk, int32_t* out_idx, float* out_score,
                                               int n_keys, Control* ctl) {
  const int n = next_pow2(count < 2 ? 2 : count);
  for (int i = count + threadIdx.x; i < n; i += blockDim.x) sel[i] = 0ull;
  __syncthreads();
  bitonic_sort_desc(sel, n, threadIdx.x, blockDim.x);
  for (int j = threadIdx.x; j < topk; j += blockDim.x) {
    bool have = j < count;
    if (have && !LT_IN_BOUNDS(key_index(sel[j]) >= 0 && key_index(sel[j]) < n_keys, ctl)) have = false;  // never publish an index outside the keys
    out_idx[j] = have ? key_index(sel[j]) : -1;
    if (out_score != nullptr) out_score[j] = have ? key_score(sel[j]) : -INFINITY;
  }
}

// ---------------------------------------------------------------------------------------------
// Keeps the `keep` largest of the `count` distinct 64-bit keys in sel[0 .. count), compacted to sel[0 .. keep)
// in any order.  MSB radix select, 8 bits per pass, histogram in shared memory (hist: 256 counters, scratch: one
// counter); the digit of each pass is found by a warp suffix scan.  Called by every thread of the CTA.
// ---------------------------------------------------------------------------------------------
constexpr int kKeepPerThread = 8;  // keys a thread holds in registers per compaction slab
__device__ __forceinline__ void keep_top_keys(uint64_t* sel, int count, int keep, unsigned int* hist, unsigned int* scratch) {
  __shared__ uint64_t s_prefix64;
  __shared__ unsigned int s_need;
  __shared__ int s_settled;
  const int tid = threadIdx.x, lane = tid & 31, nthreads = blockDim.x;
  if (tid == 0) {
    s_prefix64 = 0;
    s_need = static_cast<unsigned int>(keep);
    s_settled = 0;
  }
  uint64_t mask = 0;
  for (int pass = 0; pass < 8; ++pass) {
    const int shift = 56 - 8 * pass;
    if (tid < 256) hist[tid] = 0;
    __syncthreads();
    const uint64_t prefix = s_prefix64;
    for (int i = tid; i < count; i += nthreads) {
      const uint64_t key = sel[i];
      if ((key & mask) == prefix) atomicAdd(&hist[static_cast<unsigned int>(key >> shift) & 255u], 1u);
    }
    __syncthreads();
    if (tid < 32) {
      // suffix sums over the 256 digits, 8 per lane: the digit where the count from the top reaches `need`
      unsigned int c[8], mine = 0;
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        c[j] = hist[lane * 8 + j];
        mine += c[j];
      }
      unsigned int incl = mine;
#pragma unroll
      for (int d = 1; d < 32; d <<= 1) {
        const unsigned int o = __shfl_down_sync(0xffffffffu, incl, d);
        if (lane + d < 32) incl += o;
      }
      const unsigned int above = incl - mine, need = s_need;
      if (above < need && incl >= need) {  // exactly one lane
        unsigned int cum = above;
        for (int j = 7; j >= 0; --j) {
          if (cum + c[j] >= need) {
            s_prefix64 = prefix | (static_cast<uint64_t>(lane * 8 + j) << shift);
            s_need = need - cum;
            // every key with this prefix is wanted: the prefix padded with zeros already separates kept from
            // dropped keys, the remaining digits need no pass (the usual case once the score bytes are through)
            if (c[j] == need - cum) s_settled = 1;
            break;
          }
          cum += c[j];
        }
      }
    }
    mask |= 0xffull << shift;
    __syncthreads();
    if (s_settled) break;
  }
  const uint64_t kth = s_prefix64;  // the keep-th largest key, or a lower bound of it that no dropped key reaches
  // compaction in place, a slab of kKeepPerThread * nthreads keys at a time: every thread pulls its keys of
  // the slab into registers, then the kept ones are written from the front (never past what has been read)
  if (tid == 0) *scratch = 0;
  for (int slab = 0; slab < count; slab += kKeepPerThread * nthreads) {
    uint64_t mine[kKeepPerThread];
#pragma unroll
    for (int j = 0; j < kKeepPerThread; ++j) {
      const int i = slab + j * nthreads + tid;
      mine[j] = i < count ? sel[i] : 0ull;
    }
    __syncthreads();
#pragma unroll
    for (int j = 0; j < kKeepPerThread; ++j) {
      const int i = slab + j * nthreads + tid;
      const bool take = i < count && mine[j] >= kth;
      const unsigned int ballot = __ballot_sync(0xffffffffu, take);
      if (ballot != 0) {
        unsigned int base = 0;
        if (lane == 0) base = atomicAdd(scratch, static_cast<unsigned int>(__popc(ballot)));
        base = __shfl_sync(0xffffffffu, base, 0);
        if (take) sel[base + __popc(ballot & ((1u << lane) - 1u))] = mine[j];
      }
    }
    __syncthreads();
  }
}

// ---------------------------------------------------------------------------------------------
// final select over one row's candidate buffer (paper Sec. 3.2 "Top-k Selection").  Every candidate buffer that did not
// overflow holds the row's whole top-k, so the distribution sort takes all of its candidates.  The rows it gives up
// on go the longer way: the final threshold bin is the highest bin whose cumulative count from the top reaches k;
// every candidate at or above its lower edge is pulled into shared memory (the bins above hold fewer than k of
// them), cut to k by a radix select, sorted, and written out.
// ---------------------------------------------------------------------------------------------
template <int kFinalThreads>
__global__ void __launch_bounds__(kFinalThreads, kFinalThreads == 512 ? 3 : 1) final_select_kernel(const FinalSelectParams p, int sel_cap) {
  extern __shared__ __align__(16) uint64_t sel[];  // sel_cap keys; the distribution sort's bins are the last of them
  __shared__ unsigned int hist[kBins];
  __shared__ int s_tb;
  __shared__ unsigned int s_count;
  const int t = blockIdx.x;
  const int lane = threadIdx.x & 31;
  const uint2* cand = p.cand + static_cast<size_t>(t) * p.cap;
  chain_wait();
  // The candidates are fetched without waiting for their number: most rows have between 1 and 2 topk of them.
  uint2 first[kFineBatch];
  const int ahead = min(p.cap, 2 * p.topk);
#pragma unroll
  for (int j = 0; j < kFineBatch; ++j) {
    const int i = j * kFinalThreads + threadIdx.x;
    if (i < ahead) first[j] = __ldcs(cand + i);
  }
  const unsigned int tail = p.tail[t];
  const int vis = visible_keys(t, p.N, p.causal_offset);
  const int kk = p.topk < vis ? p.topk : vis;
  bool redo = tail > static_cast<unsigned int>(p.cap) || tail < static_cast<unsigned int>(kk);
  if (threadIdx.x == 0) {
    atomicMax(&p.ctl->max_survivors, static_cast<int>(tail > 0x7fffffffu ? 0x7fffffffu : tail));
    atomicAdd(&p.ctl->tot_survivors, static_cast<int>(tail > 0x000fffffu ? 0x000fffffu : tail));
    if (tail > static_cast<unsigned int>(p.cap)) atomicAdd(&p.ctl->overflow_rows, 1);
  }
  int32_t* out_idx = p.out_idx + static_cast<size_t>(t) * p.topk;
  float* out_score = p.out_score ? p.out_score + static_cast<size_t>(t) * p.topk : nullptr;
  if (!redo && kk > 0) {
#pragma unroll
    for (int j = 0; j < kFineBatch; ++j) {
      const int i = j * kFinalThreads + threadIdx.x;
      if (i >= ahead && i < static_cast<int>(tail)) first[j] = __ldcs(cand + i);
    }
    constexpr int kBinSlots = kFineBins * 4 / 8;
    if (fine_select_sort<kFinalThreads>([&](unsigned int i) { return __ldcs(cand + i); }, first, tail, kk, p.topk, sel,
                                        static_cast<unsigned int>(sel_cap - kBinSlots),
                                        reinterpret_cast<unsigned int*>(sel + sel_cap - kBinSlots), out_idx, out_score, p.N, p.ctl))
      return;
  }
  if (!redo) {
    // candidates are fetched eight rounds at a time so that the loads of a batch overlap; the first batch is
    // issued before the histogram work, which does not depend on it
    constexpr int kBatch = 8;
    const unsigned int rounds = (tail + kFinalThreads - 1) / kFinalThreads;
    uint2 c[kBatch];
#pragma unroll
    for (int j = 0; j < kBatch; ++j) {
      const unsigned int i = j * kFinalThreads + threadIdx.x;
      c[j] = (i < tail) ? __ldcs(cand + i) : make_uint2(0xff800000u, 0u);  // -inf never passes a finite edge
    }
    if (threadIdx.x < kBins) hist[threadIdx.x] = p.hist[static_cast<size_t>(t) * kBins + threadIdx.x];
    if (threadIdx.x == 0) s_count = 0;
    __syncthreads();
    if (threadIdx.x < 32) {
      // suffix sums over the 256 bins, 8 bins per lane, exactly as the refresh warp of the scan does
      unsigned int c[8];
      unsigned int mine = 0;
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        c[j] = hist[lane * 8 + j];
        mine += c[j];
      }
      unsigned int incl = mine;
#pragma unroll
      for (int d = 1; d < 32; d <<= 1) {
        unsigned int o = __shfl_down_sync(0xffffffffu, incl, d);
        if (lane + d < 32) incl += o;
      }
      const unsigned int above = incl - mine;
      const unsigned int need = static_cast<unsigned int>(kk);
      int tb = 0;
      if (above < need && incl >= need) {
        unsigned int cum = above;
        for (int j = 7; j >= 0; --j) {
          cum += c[j];
          if (cum >= need) {
            tb = lane * 8 + j;
            break;
          }
        }
      }
      // bin 0 is "everything else": a crossing inside lane 0 may legitimately report bin 0
      tb = __reduce_max_sync(0xffffffffu, tb);
      if (need == 0) tb = kBins - 1;
      if (lane == 0) s_tb = tb;
    }
    __syncthreads();
    const float smin = p.smin[t], width = p.width[t];
    const float edge = bin_edge(s_tb, smin, width);
    // every candidate at or above `from` goes to sel[] (one shared-memory atomic per warp); candidates beyond
    // sel_cap are counted but not stored
    auto gather = [&](float from, bool first_batch_loaded) {
      for (unsigned int r0 = 0; r0 < rounds; r0 += kBatch) {
        if (r0 > 0 || !first_batch_loaded) {
#pragma unroll
          for (int j = 0; j < kBatch; ++j) {
            const unsigned int i = (r0 + j) * kFinalThreads + threadIdx.x;
            c[j] = (i < tail) ? __ldcs(cand + i) : make_uint2(0xff800000u, 0u);
          }
        }
#pragma unroll
        for (int j = 0; j < kBatch; ++j) {
          const unsigned int i = (r0 + j) * kFinalThreads + threadIdx.x;
          const bool take = (i < tail) && (__uint_as_float(c[j].x) >= from);
          const unsigned int ballot = __ballot_sync(0xffffffffu, take);
          if (ballot != 0) {
            unsigned int base = 0;
            if (lane == 0) base = atomicAdd(&s_count, static_cast<unsigned int>(__popc(ballot)));
            base = __shfl_sync(0xffffffffu, base, 0);
            if (take) {
              const unsigned int pos = base + __popc(ballot & ((1u << lane) - 1u));
              if (pos < static_cast<unsigned int>(sel_cap)) sel[pos] = pack_key(__uint_as_float(c[j].x), static_cast<int>(c[j].y));
            }
          }
        }
      }
    };
    gather(edge, true);
    __syncthreads();
    unsigned int count = s_count;
    if (count > static_cast<unsigned int>(sel_cap) && s_tb >= 1 && s_tb < kBins - 1) {
      // The threshold bin alone holds more candidates than shared memory takes: equal-width bins over a range that
      // a few outliers stretch put most keys into a few bins (heavy-tailed scores).  Second level of the same
      // scheme inside that bin: kBins equal-width bins over [E(tb), E(tb + 1)), the bin in which the count from the
      // top reaches k, and a second gather from its lower edge.  Costs two more sweeps over the row's candidates
      // and spares the row the unfused fallback.
      const int tb = s_tb;
      const float lo = edge, hi = bin_edge(tb + 1, smin, width);
      const float w2 = (hi - lo) / static_cast<float>(kBins);
      if (w2 > 0.f) {
        __shared__ unsigned int fine[kBins];
        __shared__ unsigned int s_above;
        __shared__ float s_from;
        if (threadIdx.x < kBins) fine[threadIdx.x] = 0u;
        if (threadIdx.x < 32) {
          unsigned int above = 0;
          for (int b = tb + 1 + lane; b < kBins; b += 32) above += hist[b];
          above = __reduce_add_sync(0xffffffffu, above);
          if (lane == 0) {
            s_above = above;
            s_count = 0;
          }
        }
        __syncthreads();
        const float inv_w2 = 1.f / w2;
        for (unsigned int i = threadIdx.x; i < tail; i += kFinalThreads) {
          const float v = __uint_as_float(__ldg(&cand[i].x));
          if (v >= lo && v < hi) atomicAdd(&fine[bin_of(v, lo, w2, inv_w2)], 1u);
        }
        __syncthreads();
        if (threadIdx.x < 32) {
          // the fine bin in which the count from the top (bins above tb included) reaches kk
          unsigned int cf[8], mine = 0;
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            cf[j] = fine[lane * 8 + j];
            mine += cf[j];
          }
          unsigned int incl = mine;
#pragma unroll
          for (int d = 1; d < 32; d <<= 1) {
            const unsigned int o = __shfl_down_sync(0xffffffffu, incl, d);
            if (lane + d < 32) incl += o;
          }
          const unsigned int need = static_cast<unsigned int>(kk) - s_above;  // >= 1: bins above tb hold fewer than kk
          const unsigned int above = incl - mine;
          int fb = 0;
          if (above < need && incl >= need) {
            unsigned int cum = above;
            for (int j = 7; j >= 0; --j) {
              cum += cf[j];
              if (cum >= need) {
                fb = lane * 8 + j;
                break;
              }
            }
          }
          fb = __reduce_max_sync(0xffffffffu, fb);
          // fine bin 0 starts at the coarse edge itself: nothing gained, the row is redone
          if (lane == 0) s_from = fb >= 1 ? fminf(bin_edge(fb, lo, w2), hi) : lo;
        }
        __syncthreads();
        if (s_from > lo) {
          gather(s_from, false);
          __syncthreads();
          count = s_count;
        }
      }
    }
    // count < kk cannot happen for an exact filter; treating it as "redo" keeps the result exact regardless
    if (count > static_cast<unsigned int>(sel_cap) || count < static_cast<unsigned int>(kk)) redo = true;
    if (!redo) {
      int n_keep = static_cast<int>(count);
      if (n_keep > kk && kk > 0) {
        // More candidates than outputs.  The packed keys are distinct (the index is part of them), so the kk-th
        // largest key is unique: find it by a radix select in shared memory and keep exactly the keys at or above it.
        keep_top_keys(sel, n_keep, kk, hist, &s_count);
        n_keep = kk;
      }
      sort_and_write(sel, n_keep, p.topk, out_idx, out_score, p.N, p.ctl);
      return;
    }
  }
  if (threadIdx.x == 0) {
    p.row_flag[t] = 1;
    atomicOr(&p.ctl->status, LT_STATUS_FALLBACK);
    atomicAdd(&p.ctl->fb_rows, 1);
    if (atomicExch(p.block_flag + t / p.rows_per_block, 1u) == 0u) {
      int pos = atomicAdd(&p.ctl->fb_blocks, 1);
      p.fb_list[pos] = t / p.rows_per_block;
    }
  }
}

// ---------------------------------------------------------------------------------------------
// The kk (<= vis) best of row[0 .. vis), by one CTA, whatever bits the row holds: 4-pass MSB radix select for the kk-th score, then
// everything above it and the lowest indices among its equals, as packed keys in sel[0 .. kk), in no particular order.
// ---------------------------------------------------------------------------------------------
template <int kThreads>
__device__ __forceinline__ void radix_select_row(const float* row, int vis, int kk, uint64_t* sel, bool nan_last) {
  constexpr int kWarps = kThreads / 32;
  __shared__ unsigned int hist[256];
  __shared__ unsigned int s_prefix, s_remaining, s_gt;
  __shared__ unsigned int warp_cnt[kWarps];
  __shared__ int s_nan;
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  // NaN scores below everything, -inf included, where the row has enough others.  They are told by their bits: a test of the float
  // (isnan) next to the selection of its bits came out of nvcc 12.9 as if drop_nan were always set.
  constexpr unsigned int kLowest = 0x007fffffu, kRange = 0xff800000u - kLowest;  // ordered bit patterns of -inf .. +inf
  bool drop_nan = false;
  if (nan_last) {
    if (tid == 0) s_nan = 0;
    __syncthreads();
    int n = 0;
    for (int i = tid; i < vis; i += kThreads) n += score_to_key(__float_as_uint(row[i])) - kLowest > kRange ? 1 : 0;
    n = __reduce_add_sync(0xffffffffu, n);
    if (lane == 0 && n > 0) atomicAdd(&s_nan, n);
    __syncthreads();
    drop_nan = vis - s_nan >= kk;
  }
  const unsigned int key_lo = drop_nan ? kLowest : 0u, key_range = drop_nan ? kRange : 0xffffffffu;
  auto key_of = [&](float v) {
    const unsigned int k = score_to_key(__float_as_uint(v));
    return k - key_lo > key_range ? 0u : k;
  };
  if (tid == 0) {
    s_prefix = 0;
    s_remaining = static_cast<unsigned int>(kk);
  }
  unsigned int mask = 0;
  for (int pass = 0; pass < 4; ++pass) {
    const int shift = 24 - 8 * pass;
    if (tid < 256) hist[tid] = 0;
    __syncthreads();
    const unsigned int prefix = s_prefix;
    // Scores of one row share their leading bits, so consecutive candidates of a thread mostly want the
    // same counter: each thread run-length-encodes its digits and issues one atomic per run.
    unsigned int run_digit = 0x100u, run_len = 0;
    // (kSelBatch loads in flight per thread: one row is read by one SM, which is latency-bound otherwise)
    for (int base = 0; base < vis; base += kThreads * kSelBatch) {
      float v[kSelBatch];
#pragma unroll
      for (int j = 0; j < kSelBatch; ++j) {
        const int i = base + j * kThreads + tid;
        v[j] = i < vis ? row[i] : 0.f;
      }
#pragma unroll
      for (int j = 0; j < kSelBatch; ++j) {
        const int i = base + j * kThreads + tid;
        unsigned int digit = 0x100u;  // "not a candidate" (out of range or another prefix)
        if (i < vis) {
          const unsigned int key = key_of(v[j]);
          if ((key & mask) == prefix) digit = (key >> shift) & 255u;
        }
        if (digit < 0x100u) {
          if (digit == run_digit) {
            ++run_len;
          } else {
            if (run_len > 0) atomicAdd(&hist[run_digit], run_len);
            run_digit = digit;
            run_len = 1;
          }
        }
      }
    }
    if (run_len > 0) atomicAdd(&hist[run_digit], run_len);
    __syncthreads();
    if (tid < 32) {
      // suffix sums over the 256 digits, 8 per lane: the digit where the count from the top reaches what is still needed
      unsigned int c[8], mine = 0;
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        c[j] = hist[lane * 8 + j];
        mine += c[j];
      }
      unsigned int incl = mine;
#pragma unroll
      for (int d = 1; d < 32; d <<= 1) {
        const unsigned int o = __shfl_down_sync(0xffffffffu, incl, d);
        if (lane + d < 32) incl += o;
      }
      const unsigned int remaining = s_remaining;
      unsigned int cum = incl - mine;
      __syncwarp();
      if (cum < remaining && incl >= remaining) {  // exactly one lane
        int digit = -1;
#pragma unroll
        for (int j = 7; j >= 0; --j) {
          if (digit < 0 && cum + c[j] >= remaining) digit = lane * 8 + j;
          if (digit < 0) cum += c[j];
        }
        s_remaining = remaining - cum;  // still needed among keys that share the longer prefix
        s_prefix = prefix | (static_cast<unsigned int>(digit) << shift);
      }
    }
    mask |= 0xffu << shift;
    __syncthreads();
  }
  const unsigned int kth = s_prefix;                 // key of the k-th largest score
  const unsigned int need_eq = s_remaining;          // how many keys equal to it are selected
  const unsigned int n_gt = static_cast<unsigned int>(kk) - need_eq;
  if (tid == 0) s_gt = 0;
  // Collection.  Keys above the k-th go in any order (the sort follows).  Ties at the k-th value keep
  // the lowest indices, so they are ranked in index order: every warp owns one contiguous range of the
  // row, counts its ties, and after one prefix sum over the warps writes them at their ranks.
  const int per_warp = (((vis + kWarps - 1) / kWarps + 31) / 32) * 32;  // range length: a multiple of 32 covering vis / kWarps
  const int lo = wid * per_warp;
  const int hi = min(vis, lo + per_warp);
  unsigned int my_eq = 0;
  for (int base = lo; base < hi; base += 32 * kSelBatch) {
    float v[kSelBatch];
#pragma unroll
    for (int j = 0; j < kSelBatch; ++j) {
      const int i = base + j * 32 + lane;
      v[j] = i < hi ? row[i] : 0.f;
    }
#pragma unroll
    for (int j = 0; j < kSelBatch; ++j) {
      const int i = base + j * 32 + lane;
      const bool eq = i < hi && key_of(v[j]) == kth;
      my_eq += __popc(__ballot_sync(0xffffffffu, eq));
    }
  }
  if (lane == 0) warp_cnt[wid] = my_eq;
  __syncthreads();
  unsigned int running = 0;
  for (int wq = 0; wq < wid; ++wq) running += warp_cnt[wq];
  for (int base0 = lo; base0 < hi; base0 += 32 * kSelBatch) {
   float v[kSelBatch];
#pragma unroll
   for (int j = 0; j < kSelBatch; ++j) {
     const int i = base0 + j * 32 + lane;
     v[j] = i < hi ? row[i] : 0.f;
   }
#pragma unroll
   for (int j = 0; j < kSelBatch; ++j) {
    const int i = base0 + j * 32 + lane;
    unsigned int key = 0;
    bool gt = false, eq = false;
    if (i < hi) {
      key = key_of(v[j]);
      gt = key > kth;
      eq = key == kth;
    }
    const uint64_t packed = (static_cast<uint64_t>(key) << 32) | (0xffffffffu - static_cast<unsigned int>(i));
    const unsigned int gt_ballot = __ballot_sync(0xffffffffu, gt);
    if (gt_ballot != 0) {
      unsigned int pos = 0;
      if (lane == 0) pos = atomicAdd(&s_gt, static_cast<unsigned int>(__popc(gt_ballot)));
      pos = __shfl_sync(0xffffffffu, pos, 0);
      if (gt) sel[pos + __popc(gt_ballot & ((1u << lane) - 1u))] = packed;
    }
    const unsigned int eq_ballot = __ballot_sync(0xffffffffu, eq);
    if (eq) {
      const unsigned int rank = running + __popc(eq_ballot & ((1u << lane) - 1u));
      if (rank < need_eq) sel[n_gt + rank] = packed;
    }
    running += __popc(eq_ballot);
   }
  }
}

// ---------------------------------------------------------------------------------------------
// full-row exact select.  A row of at most kSelDirect visible keys goes straight through the distribution sort; a longer
// one (or one with mass ties) takes a 4-pass MSB radix select for the k-th key, ordered collection of ties (lowest
// indices first), and a sort of the k winners.
// ---------------------------------------------------------------------------------------------
template <int kThreads, bool kInLoop>
__device__ __forceinline__ void select_one_row(const SelectRowsParams& p, int t, const float* row, int slot) {
  extern __shared__ __align__(16) uint64_t sel_smem[];  // the distribution sort's bins, then two buffers of p.sel_slots keys
  unsigned int* bins = reinterpret_cast<unsigned int*>(sel_smem);
  uint64_t* sel = sel_smem + kFineBins * 4 / 8;
  const int vis = visible_keys(t, p.N, p.causal_offset);
  const int kk = p.topk < vis ? p.topk : vis;
  int32_t* out_idx = p.out_idx + static_cast<size_t>(t) * p.topk;
  float* out_score = p.out_score ? p.out_score + static_cast<size_t>(t) * p.topk : nullptr;
  const int tid = threadIdx.x;

  if (vis == 0) {
    add_status(p.ctl, slot);
    sort_and_write(sel, 0, p.topk, out_idx, out_score, p.N, p.ctl);
    return;
  }
  uint2 first[kFineBatch];
  if (vis <= kSelDirect) {
#pragma unroll
    for (int j = 0; j < kFineBatch; ++j) {
      const int i = j * kThreads + tid;
      if (i < vis) first[j] = make_uint2(__float_as_uint(row[i]), static_cast<unsigned int>(i));
    }
    add_status(p.ctl, slot);
    if (fine_select_sort<kThreads, kInLoop>([&](unsigned int i) { return make_uint2(__float_as_uint(row[i]), i); }, first,
                                      static_cast<unsigned int>(vis), kk, p.topk, sel, 2u * p.sel_slots, bins, out_idx, out_score,
                                      p.N, p.ctl, p.nan_last != 0 && vis > p.topk))
      return;
  }
  if (vis <= p.topk) {
    if (vis > kSelDirect) add_status(p.ctl, slot);
    // every visible key is selected, and they did not spread over the bins
    for (int i = tid; i < vis; i += kThreads) sel[i] = pack_key(row[i], i);
    __syncthreads();
    sort_and_write(sel, vis, p.topk, out_idx, out_score, p.N, p.ctl);
    return;
  }

  if (vis > kSelDirect) add_status(p.ctl, slot);
  radix_select_row<kThreads>(row, vis, kk, sel, p.nan_last != 0);
  __syncthreads();
  auto winner = [&](unsigned int i) { return make_uint2(key_to_score_bits(static_cast<unsigned int>(sel[i] >> 32)), static_cast<unsigned int>(key_index(sel[i]))); };
#pragma unroll
  for (int j = 0; j < kFineBatch; ++j)
    if (j * kThreads + tid < kk) first[j] = winner(j * kThreads + tid);
  if (fine_select_sort<kThreads, kInLoop>(winner, first, static_cast<unsigned int>(kk), kk, p.topk, sel + p.sel_slots, p.sel_slots, bins,
                                 out_idx, out_score, p.N, p.ctl))
    return;
  sort_and_write(sel, kk, p.topk, out_idx, out_score, p.N, p.ctl);
}

// kFlagged: the rows that row_flag marks (the exact fallback).  They are few or none, and only the device knows: a grid of at most
// two CTAs for every SM goes through all of them.  (A CTA per row took 21 us, with the scan ahead of it, to find nothing to do among 4096 rows and 39 us, in two rounds, among 8192; now 9 and 12.)
// (The row's select is out of line there: inlined into the loop, 4 rows of 2^20 keys through the fallback 1.20 ms, so 1.08; a CTA per row 1.17.
// Whole calls with every row flagged, a CTA per row / now: 8 x 16 K 36.0 / 35.1 us, 148 x 8 K 64.8 / 64.2, 4096 x 8 K 939 / 886.)
template <int kThreads>
__device__ __noinline__ void select_flagged_row(const SelectRowsParams& p, int t, const float* row) {
  select_one_row<kThreads, true>(p, t, row, 0);
}
template <int kThreads, bool kFlagged>
__global__ void __launch_bounds__(kThreads, kThreads <= 512 ? 3 : 1) select_rows_kernel(const __grid_constant__ SelectRowsParams p) {
  chain_wait();
  if (!kFlagged) {  // a CTA for every row
    const int slot = load_status_slot(p.status_slots, p.n_slots, threadIdx.x, p.ctl);
    select_one_row<kThreads, false>(p, p.row_begin + blockIdx.x, p.scores + static_cast<size_t>(blockIdx.x) * p.ld, slot);
    return;
  }
  const int n = p.fb_list != nullptr ? min(p.n_blocks, (*p.fb_blocks - p.fb_round_base) * p.rows_per_block) : p.n_blocks;
  for (int b = blockIdx.x; b < n; b += gridDim.x) {
    const int t = p.fb_list != nullptr ? p.fb_list[p.fb_round_base + b / p.rows_per_block] * p.rows_per_block + b % p.rows_per_block : p.row_begin + b;
    if (t >= p.T || !p.row_flag[t]) continue;
    __syncthreads();  // the row before is done with the shared memory
    select_flagged_row<kThreads>(p, t, p.scores + static_cast<size_t>(b) * p.ld);
  }
}

// ---------------------------------------------------------------------------------------------
// Full-row exact select by a cluster of CTAs, for few rows over many keys (one CTA would stream a 128 K row three to
// four times on its own).  Every CTA owns a slice of the row, kept in shared memory as far as it fits.  Equal-width
// bins over the row's range, as in the distribution sort but kClBins of them: the CTAs' histograms are merged through
// distributed shared memory, the CTAs agree on the bin that holds the kk-th key, and every key up to it goes to the
// first CTA's list, which is then sorted there.  A bin that holds more keys than the list takes is split again over
// its own range (a few outliers stretch the range), and a bin of one single value by the keys' indices, in whose order ties
// are taken (1 x 300 K keys of 50 different scores, topk 64: 453 us when the row was left to a radix select by one CTA, now 42);
// what still does not fit, and a row with infinite or NaN scores
// or with whatever a scan that gave up left behind, goes to the first CTA's radix select over the whole row, which is total.  Bound by latencies (four cluster barriers, a sort by one CTA) up to 128 K keys, by
// instructions above: a key costs about 15, on floats throughout (ordered bit patterns would double that).
// ---------------------------------------------------------------------------------------------
constexpr int kClThreads = 512;
constexpr int kClWarps = kClThreads / 32;
constexpr int kClBins = 2048;
constexpr int kClLevels = 6;  // ties next to a dense stretch of scores (ReLU's exact zeros) take one more for every factor of 2048
constexpr int kClStaticSmem = 8 * 1024;  // upper bound of what the kernel declares statically
// (a multiple of four keys: what lies behind the list is accessed in 16-byte pieces)
__host__ __device__ constexpr int cluster_list_cap(int topk) { return (topk + (topk / 4 > 2048 ? topk / 4 : 2048) + 3) / 4 * 4; }

__device__ __forceinline__ unsigned int warp_inclusive_sum(unsigned int v, int lane) {
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const unsigned int o = __shfl_up_sync(0xffffffffu, v, d);
    if (lane >= d) v += o;
  }
  return v;
}

// The rare ways of the cluster select are out of line: it lives for a few microseconds, and its usual way is shorter without them (1 x
// 32 K dense, topk 2048, 20.9 -> 20.4 us).  (Inlined into the select by one CTA, the radix select costs nothing.)
__device__ __noinline__ void radix_select_row_rare(const float* row, int vis, int kk, uint64_t* sel, bool nan_last) {
  radix_select_row<kClThreads>(row, vis, kk, sel, nan_last);
}

// A threshold bin of one value.  A CTA's slice in pieces of four: the first n_held from shared memory.
__device__ __forceinline__ int tied_shift(int vis) { return 32 - __clz(static_cast<unsigned int>(vis - 1) / kClBins); }
struct TiedSlice {
  const float4* held;
  const float4* rest;
  int n_held, n, lo, len, shift;
  float value;
  template <class Visit>
  __device__ __forceinline__ void sweep(Visit&& visit) const {  // visit(score, index in the row)
    for (int i = threadIdx.x; i < n; i += kClThreads) {
      const float4 v = i < n_held ? held[i] : __ldcg(rest + i);
      visit(v.x, lo + 4 * i);
      if (4 * i + 1 < len) visit(v.y, lo + 4 * i + 1);
      if (4 * i + 2 < len) visit(v.z, lo + 4 * i + 2);
      if (4 * i + 3 < len) visit(v.w, lo + 4 * i + 3);
    }
  }
};
// bins[b] = ties among the keys of run b (2^shift consecutive keys of the row)
__device__ __noinline__ void count_tied(const TiedSlice t, unsigned int* bins) {
  t.sweep([&](float v, int i) {
    if (v == t.value) atomicAdd(&bins[i >> t.shift], 1u);
  });
}
// every key above the ties, and the ties of the runs up to last_run, to the list; *fill counts it
__device__ __noinline__ void collect_tied(const TiedSlice t, int last_run, uint64_t* list, unsigned int* fill) {
  t.sweep([&](float v, int i) {
    if (v > t.value || (v == t.value && (i >> t.shift) <= last_run)) list[atomicAdd(fill, 1u)] = pack_key(v, i);
  });
}

// p.slice_keys: scores of a slice kept in shared memory (a multiple of 4).  kPerSm: CTAs to an SM the registers are cut for: one while
// clusters find free SMs easily (up to 64 CTAs: no spills, 16 x 32 K 25.2 -> 24.4 us), two beyond (128 CTAs in clusters of 8: 16 x
// 100 K 40.3 -> 35.3 us).
template <int kPerSm>
__global__ void __launch_bounds__(kClThreads, kPerSm) select_cluster_kernel(const SelectRowsParams p) {
  namespace cg = cooperative_groups;
  cg::cluster_group cl = cg::this_cluster();
  const unsigned int n_cta = cl.num_blocks(), rank = cl.block_rank();
  extern __shared__ __align__(16) uint8_t cl_smem[];
  const unsigned int cap = static_cast<unsigned int>(cluster_list_cap(p.topk));
  uint64_t* list = reinterpret_cast<uint64_t*>(cl_smem);             // keys up to the threshold bin (first CTA)
  unsigned int* bins = reinterpret_cast<unsigned int*>(list + cap);  // this CTA's histogram; later the sort's bins
  float* slice = reinterpret_cast<float*>(bins + kFineBins);
  uint64_t* sorted = reinterpret_cast<uint64_t*>(slice);             // the slice is dead when the list is sorted
  __shared__ __align__(16) unsigned int s_seg[kClBins / 2];
  __shared__ float s_range[2], s_wmin[kClWarps], s_wmax[kClWarps];
  __shared__ unsigned int s_sum[kClWarps], s_seg_sum, s_count, s_above, s_tb, s_total, s_fill;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int t = p.row_begin + blockIdx.x / n_cta;
  const float* row = p.scores + static_cast<size_t>(t - p.row_begin) * p.ld;
  const int vis = visible_keys(t, p.N, p.causal_offset);
  const int kk = p.topk < vis ? p.topk : vis;
  int32_t* out_idx = p.out_idx + static_cast<size_t>(t) * p.topk;
  float* out_score = p.out_score ? p.out_score + static_cast<size_t>(t) * p.topk : nullptr;
  chain_wait();
  const int slot = load_status_slot(p.status_slots, p.n_slots, tid, p.ctl);
  if (kk == 0) {  // the whole cluster
    add_status(p.ctl, slot);
    if (rank == 0) sort_and_write(list, 0, p.topk, out_idx, out_score, p.N, p.ctl);
    return;
  }
  // slices start on 16-byte boundaries (the caller's rows do); the last of a slice's pieces of four may be ragged
  const int per = ((vis + static_cast<int>(n_cta) - 1) / static_cast<int>(n_cta) + 3) & ~3;
  const int lo = min(vis, static_cast<int>(rank) * per), len = min(vis, lo + per) - lo;
  const int held = min(len, p.slice_keys);
  const float4* mine4 = reinterpret_cast<const float4*>(row + lo);
  float4* slice4 = reinterpret_cast<float4*>(slice);
  constexpr int kDepth = 8;
  // pieces [from, to) of the slice from global memory, kDepth of them in flight; visit(piece number, values)
  auto stream = [&](int from, int to, auto&& visit) {
    for (int base = from + tid; base < to; base += kDepth * kClThreads) {
      float4 v[kDepth];
#pragma unroll
      for (int j = 0; j < kDepth; ++j) v[j] = __ldcg(mine4 + min(base + j * kClThreads, to - 1));
#pragma unroll
      for (int j = 0; j < kDepth; ++j)
        if (base + j * kClThreads < to) visit(base + j * kClThreads, v[j]);
    }
  };
  const int pieces = (len + 3) >> 2, held_pieces = held >= len ? pieces : held >> 2;
  // visits (score, index in the slice) of every key of the slice.  A ragged last piece was padded with -inf when it was
  // loaded; -inf lies below every range and is never counted or taken.
  const float kNone = -INFINITY;
  auto clip = [&](int piece, float4 v) {
    if (piece * 4 + 3 >= len) {
      if (piece * 4 + 1 >= len) v.y = kNone;
      if (piece * 4 + 2 >= len) v.z = kNone;
      v.w = kNone;
    }
    return v;
  };
  auto sweep = [&](auto&& visit) {
#pragma unroll 2
    for (int i = tid; i < held_pieces; i += kClThreads) visit(i, slice4[i]);
    stream(held_pieces, pieces, [&](int i, float4 v) { visit(i, clip(i, v)); });
  };
  float vmin = INFINITY, vmax = -INFINITY;
  stream(0, pieces, [&](int i, float4 v) {
    float4 m = v;  // for the minimum, padding repeats a real score (v.x always is one)
    if (i * 4 + 3 >= len) {
      v = clip(i, v);
      m = make_float4(v.x, i * 4 + 1 < len ? v.y : v.x, i * 4 + 2 < len ? v.z : v.x, v.x);
    }
    if (i < held_pieces) slice4[i] = v;
    vmin = fminf(vmin, fminf(fminf(m.x, m.y), fminf(m.z, m.w)));
    vmax = fmaxf(vmax, fmaxf(fmaxf(m.x, m.y), fmaxf(m.z, m.w)));
  });
  add_status(p.ctl, slot);
  if (tid == 0) s_fill = 0u;

  float scale = 0.f, limit = 0.f;
  unsigned int above = 0u, total = 0u;
  bool tied = false;
  int level = 0;
  for (;; ++level) {
    // range [vmin, vmax] of the keys still in question, over the cluster
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) {
      vmin = fminf(vmin, __shfl_xor_sync(0xffffffffu, vmin, d));
      vmax = fmaxf(vmax, __shfl_xor_sync(0xffffffffu, vmax, d));
    }
    if (lane == 0) {
      s_wmin[warp] = vmin;
      s_wmax[warp] = vmax;
    }
    for (int i = tid; i < kClBins / 4; i += kClThreads) reinterpret_cast<uint4*>(bins)[i] = make_uint4(0u, 0u, 0u, 0u);
    __syncthreads();
    if (tid == 0) {
#pragma unroll
      for (int w = 1; w < kClWarps; ++w) {
        vmin = fminf(vmin, s_wmin[w]);
        vmax = fmaxf(vmax, s_wmax[w]);
      }
      s_range[0] = vmin;
      s_range[1] = vmax;
    }
    cl.sync();
    {
      const float* r = cl.map_shared_rank(s_range, min(static_cast<unsigned int>(lane), n_cta - 1u));
      vmin = r[0];
      vmax = r[1];
#pragma unroll
      for (int d = 16; d > 0; d >>= 1) {
        vmin = fminf(vmin, __shfl_xor_sync(0xffffffffu, vmin, d));
        vmax = fmaxf(vmax, __shfl_xor_sync(0xffffffffu, vmax, d));
      }
    }
    // Infinite scores (sums that overflowed) and ranges too wide for a float have no bins: the first CTA ranks the row's bit
    // patterns instead.  Every CTA has the same range, so all of them leave together.
    if (!(fabsf(vmax - vmin) <= FLT_MAX)) {
      total = cap + 1u;
      break;
    }
    // bin of a score in the range, best scores first; monotone because every step rounds monotonically
    // (finite, so that the best score's 0 * scale is 0)
    tied = vmax == vmin;
    scale = tied ? 0.f : fminf(static_cast<float>(kClBins) / (vmax - vmin), 3e38f);
    auto count = [&](float v) {
      if (v >= vmin && v <= vmax) atomicAdd(&bins[min(static_cast<unsigned int>((vmax - v) * scale), kClBins - 1u)], 1u);
    };
    if (tied) {
      count_tied(TiedSlice{slice4, mine4, held_pieces, pieces, lo, len, tied_shift(vis), vmax}, bins);
    } else {
      sweep([&](int, float4 v) {
        count(v.x);
        count(v.y);
        count(v.z);
        count(v.w);
      });
    }
    cl.sync();
    // merge: this CTA sums the bins of its segment over the cluster
    const int seg = kClBins / static_cast<int>(n_cta);  // 128 .. 1024
    unsigned int part = 0;
    for (int i = tid; i < seg; i += kClThreads) {
      unsigned int c = 0;
#pragma unroll 4
      for (unsigned int r = 0; r < n_cta; ++r) c += cl.map_shared_rank(bins, r)[rank * seg + i];
      s_seg[i] = c;
      part += c;
    }
    part = __reduce_add_sync(0xffffffffu, part);
    if (lane == 0) s_sum[warp] = part;
    __syncthreads();
    if (tid < 32) {
      part = __reduce_add_sync(0xffffffffu, lane < kClWarps ? s_sum[lane] : 0u);
      if (lane == 0) s_seg_sum = part;
    }
    cl.sync();
    {
      // the segment, then the bin in it, where the count from the top reaches kk (every warp finds the segment)
      const unsigned int need = static_cast<unsigned int>(kk) - above;
      const unsigned int sum = lane < static_cast<int>(n_cta) ? *cl.map_shared_rank(&s_seg_sum, lane) : 0u;
      const unsigned int incl = warp_inclusive_sum(sum, lane);
      const unsigned int crossing = __ballot_sync(0xffffffffu, incl >= need && incl - sum < need);
      // NaN scores are counted nowhere: as above.  (crossing is zero only where keys are missing from the counts; it is tested
      // because the address below is made from it.)
      if ((level == 0 && __shfl_sync(0xffffffffu, incl, 31) != static_cast<unsigned int>(vis)) || crossing == 0u) {
        total = cap + 1u;
        break;
      }
      const int owner = __ffs(crossing) - 1;
      const unsigned int before = __shfl_sync(0xffffffffu, incl - sum, owner);
      const uint2* segc = reinterpret_cast<const uint2*>(cl.map_shared_rank(s_seg, owner));
      const uint2 c = 2 * tid < seg ? segc[tid] : make_uint2(0u, 0u);  // two bins per thread: at most 1024
      const unsigned int ic = warp_inclusive_sum(c.x + c.y, lane);
      if (lane == 31) s_sum[warp] = ic;
      __syncthreads();
      const unsigned int at = before + __reduce_add_sync(0xffffffffu, lane < warp ? s_sum[lane] : 0u) + ic - c.x - c.y;  // keys above this thread's bins
      if (at < need && at + c.x + c.y >= need) {  // exactly one thread
        const bool second = at + c.x < need;
        s_tb = static_cast<unsigned int>(owner * seg + 2 * tid) + (second ? 1u : 0u);
        s_above = above + at + (second ? c.x : 0u);
        s_total = above + at + c.x + (second ? c.y : 0u);
      }
      __syncthreads();
    }
    const unsigned int tb = s_tb;
    total = s_total;
    // a key is wanted when it lies in the range or above it and (vmax - v) * scale < limit
    limit = tb == kClBins - 1u ? INFINITY : static_cast<float>(tb + 1u);
    if (total <= cap || tied || level == kClLevels - 1) break;
    above = s_above;
    // the threshold bin alone is the next level's range
    float nmin = INFINITY, nmax = -INFINITY;
    const float from = static_cast<float>(tb);
    auto narrow = [&](float v) {
      const float d = (vmax - v) * scale;
      if (v >= vmin && v <= vmax && d >= from && d < limit) {
        nmin = fminf(nmin, v);
        nmax = fmaxf(nmax, v);
      }
    };
    sweep([&](int, float4 v) {
      narrow(v.x);
      narrow(v.y);
      narrow(v.z);
      narrow(v.w);
    });
    vmin = nmin;
    vmax = nmax;
  }
  if (total <= cap && tied) {
    collect_tied(TiedSlice{slice4, mine4, held_pieces, pieces, lo, len, tied_shift(vis), vmax}, static_cast<int>(s_tb),
                 cl.map_shared_rank(list, 0), cl.map_shared_rank(&s_fill, 0));
  } else if (total <= cap) {
    // every wanted key to the first CTA's list: count, reserve, write
    auto wanted = [&](float v) { return v >= vmin && (vmax - v) * scale < limit; };
    unsigned int n = 0;
    sweep([&](int, float4 v) { n += (wanted(v.x) ? 1u : 0u) + (wanted(v.y) ? 1u : 0u) + (wanted(v.z) ? 1u : 0u) + (wanted(v.w) ? 1u : 0u); });
    const unsigned int incl = warp_inclusive_sum(n, lane);
    if (lane == 31) s_sum[warp] = incl;
    __syncthreads();
    if (tid < 32) {
      const unsigned int w = lane < kClWarps ? s_sum[lane] : 0u;
      const unsigned int wi = warp_inclusive_sum(w, lane);
      unsigned int base = 0;
      if (lane == 31 && wi > 0u) base = atomicAdd(cl.map_shared_rank(&s_fill, 0), wi);
      base = __shfl_sync(0xffffffffu, base, 31);
      if (lane < kClWarps) s_sum[lane] = base + wi - w;
    }
    __syncthreads();
    unsigned int pos = s_sum[warp] + incl - n;
    uint64_t* dst = cl.map_shared_rank(list, 0);
    if (n > 0u)
      sweep([&](int i, float4 v) {
        if (wanted(v.x)) dst[pos++] = pack_key(v.x, lo + 4 * i);
        if (wanted(v.y)) dst[pos++] = pack_key(v.y, lo + 4 * i + 1);
        if (wanted(v.z)) dst[pos++] = pack_key(v.z, lo + 4 * i + 2);
        if (wanted(v.w)) dst[pos++] = pack_key(v.w, lo + 4 * i + 3);
      });
  }
  cl.sync();  // the list is complete; nothing of the other CTAs is read any more
  if (rank != 0) return;
  if (total <= cap) {
    uint2 first[kFineBatch];
    auto entry = [&](unsigned int i) { return make_uint2(key_to_score_bits(static_cast<unsigned int>(list[i] >> 32)), static_cast<unsigned int>(key_index(list[i]))); };
#pragma unroll
    for (int j = 0; j < kFineBatch; ++j)
      if (j * kClThreads + tid < total) first[j] = entry(j * kClThreads + tid);
    if (fine_select_sort<kClThreads>(entry, first, total, kk, p.topk, sorted, cap, bins, out_idx, out_score, p.N, p.ctl)) return;
    if (total > static_cast<unsigned int>(kk)) keep_top_keys(list, static_cast<int>(total), kk, bins, &s_count);
  } else {
    radix_select_row_rare(row, vis, kk, list, p.nan_last != 0);
  }
  __syncthreads();
  // room for next_pow2(kk) keys: the list, the bins and the slice lie one behind the other
  sort_and_write(list, kk, p.topk, out_idx, out_score, p.N, p.ctl);
}

}  // namespace

namespace {
template <int kDtype, int kRows>
cudaError_t launch_simt_rows(const void* q, const float* w, const void* k, const float* k_scale, int N, int H, int D, int causal_offset,
                             int row_begin, int row_end, float* out, long long ld, Control* clear_ctl, cudaStream_t stream) {
  constexpr int kKeys = 128 * (8 / kRows);
  const int tiles = (N + kKeys - 1) / kKeys;
  // (at most 65,535 row blocks to a launch)
  for (int r0 = row_begin; r0 < row_end; r0 += kRows * 65535) {
    const int r1 = row_end - r0 < kRows * 65535 ? row_end : r0 + kRows * 65535;
    const cudaError_t e = launch_chained(simt_scores_kernel<kDtype, kRows>, dim3(tiles, (r1 - r0 + kRows - 1) / kRows), kSimtThreads, 0,
                                         stream, 1, q, w, k, k_scale, N, H, D, causal_offset, r0, r1,
                                         out + static_cast<size_t>(r0 - row_begin) * ld, ld, r0 == row_begin ? clear_ctl : nullptr);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}
template <int kDtype>
cudaError_t launch_simt_typed(const void* q, const float* w, const void* k, const float* k_scale, int N, int H, int D, int causal_offset,
                              int row_begin, int row_end, float* out, long long ld, Control* clear_ctl, cudaStream_t stream) {
  const int rows = row_end - row_begin;
  // a key tile is read once per kRows query rows; a few rows over many keys give the warps more keys instead
  if (rows > 4 || N <= 256 * 148) return launch_simt_rows<kDtype, 8>(q, w, k, k_scale, N, H, D, causal_offset, row_begin, row_end, out, ld, clear_ctl, stream);
  return launch_simt_rows<kDtype, 4>(q, w, k, k_scale, N, H, D, causal_offset, row_begin, row_end, out, ld, clear_ctl, stream);
}
}  // namespace

cudaError_t launch_zero(void* p, size_t bytes, cudaStream_t stream) {
  const long long n = static_cast<long long>(bytes / 16);
  if (n <= 0) return cudaSuccess;
  const long long blocks = (n + 1023) / 1024 < 592 ? (n + 1023) / 1024 : 592;
  return launch_chained(zero_kernel, static_cast<unsigned int>(blocks), 256, 0, stream, 1, static_cast<uint4*>(p), n);
}

cudaError_t launch_simt_scores(int dtype, const void* q, const float* w, const void* k, const float* k_scale, int T, int N,
                               int H, int D, int causal_offset, int row_begin, int row_end, float* out, long long ld,
                               Control* clear_ctl, cudaStream_t stream) {
  (void)T;
  if (row_end <= row_begin) return cudaSuccess;
  if (dtype == LT_DTYPE_F32) return launch_simt_typed<LT_DTYPE_F32>(q, w, k, k_scale, N, H, D, causal_offset, row_begin, row_end, out, ld, clear_ctl, stream);
  if (dtype == LT_DTYPE_BF16) return launch_simt_typed<LT_DTYPE_BF16>(q, w, k, k_scale, N, H, D, causal_offset, row_begin, row_end, out, ld, clear_ctl, stream);
  return launch_simt_typed<LT_DTYPE_E4M3>(q, w, k, k_scale, N, H, D, causal_offset, row_begin, row_end, out, ld, clear_ctl, stream);
}

cudaError_t launch_sample_stats(const float* sample, int T, int n_sample, int rank, float* smin, float* width, float* thr,
                                const OpenParams* open, cudaStream_t stream) {
  const OpenParams o = open != nullptr ? *open : OpenParams{};
  // few rows leave the chip idle: a large CTA then shortens the sweeps; with many rows small CTAs overlap better
  const bool few = T <= 2 * sm_count();
  auto launch = [&](auto kernel, int threads) { return launch_chained(kernel, T, threads, 0, stream, 1, sample, n_sample, rank, smin, width, thr, o); };
  if (n_sample < kStatsShort || static_cast<long long>(rank) * kStatsHighShare >= n_sample) return few ? launch(sample_stats_kernel<1024, 0>, 1024) : launch(sample_stats_kernel<256, 0>, 256);
  if (few) return launch(sample_stats_kernel<1024, 8>, 1024);
  if (n_sample > 4096) return launch(sample_stats_kernel<512, 16>, 512);
  return launch(sample_stats_kernel<256, 16>, 256);
}

cudaError_t launch_final_select(const FinalSelectParams& p, cudaStream_t stream) {
  // room for every candidate at or above the final threshold edge: k plus the population of the threshold bin,
  // which for a small k over millions of keys can be several thousand (the select that follows cuts them to k)
  int sel_cap = next_pow2(2 * p.topk);
  if (sel_cap < 8192) sel_cap = 8192;
  if (sel_cap > kSelCap) sel_cap = kSelCap;
  const int smem = sel_cap * static_cast<int>(sizeof(uint64_t));
  // a row to an SM gets all the threads it can use (4 rows of 6.4 k candidates 16.4 -> 10.2 us, 77 of 3.5 k 14.3 -> 10.2); more rows share
  // SMs, and small CTAs hide one another's barriers
  static std::atomic<unsigned long long> done[2];
  cudaError_t e = allow_smem(reinterpret_cast<const void*>(final_select_kernel<512>), done[0]);
  if (e == cudaSuccess) e = allow_smem(reinterpret_cast<const void*>(final_select_kernel<1024>), done[1]);
  if (e != cudaSuccess) return e;
  if (p.T <= sm_count()) return launch_chained(final_select_kernel<1024>, p.T, 1024, smem, stream, 1, p, sel_cap);
  return launch_chained(final_select_kernel<512>, p.T, 512, smem, stream, 1, p, sel_cap);
}

cudaError_t launch_select_dense(const SelectRowsParams& params, cudaStream_t stream) {
  // one CTA sorts a short row in one go; a cluster shares a longer one, as wide as the row is long and the chip allows
  if (params.N <= kSelDirect) return launch_select_rows(params, stream);
  SelectRowsParams p = params;
  if (p.n_blocks <= 0) return cudaSuccess;
  static std::atomic<unsigned long long> done[2];
  cudaError_t e = allow_smem(reinterpret_cast<const void*>(select_cluster_kernel<1>), done[0], true);
  if (e == cudaSuccess) e = allow_smem(reinterpret_cast<const void*>(select_cluster_kernel<2>), done[1], true);
  if (e != cudaSuccess) return e;
  static std::atomic<signed char> widest[64];
  const int width = select_cluster_width(p.N, p.n_blocks, widest_cluster(select_cluster_kernel<1>, kClThreads, 227 * 1024 - kClStaticSmem, widest));
  if (width < 2) return launch_select_rows(params, stream);
  // shared memory: the list, the bins, and as much of a slice as fits (at least the sort's second buffer)
  const int list = cluster_list_cap(p.topk) * 8;
  const int slice_max = (227 * 1024 - kClStaticSmem - list - kFineBins * 4) / 16 * 4;
  const int slice_want = ((p.N + width - 1) / width + 7) / 4 * 4;
  p.slice_keys = slice_want < slice_max ? slice_want : slice_max;
  const int tail = p.slice_keys * 4 > list ? p.slice_keys * 4 : list;
  const int smem = list + kFineBins * 4 + tail;
  auto kernel = static_cast<long long>(p.n_blocks) * width <= 64 ? select_cluster_kernel<1> : select_cluster_kernel<2>;
  return launch_chained(kernel, p.n_blocks * width, kClThreads, smem, stream, width, p);
}

namespace {
template <int kThreads, bool kFlagged>
cudaError_t launch_select_rows_n(const SelectRowsParams& p, int smem, cudaStream_t stream) {
  static std::atomic<unsigned long long> done{0};
  cudaError_t e = allow_smem(reinterpret_cast<const void*>(select_rows_kernel<kThreads, kFlagged>), done);
  if (e != cudaSuccess) return e;
  const int most = 2 * sm_count();
  const int ctas = kFlagged && p.n_blocks > most ? most : p.n_blocks;
  return launch_chained(select_rows_kernel<kThreads, kFlagged>, ctas, kThreads, smem, stream, 1, p);
}
}  // namespace

cudaError_t launch_select_rows(const SelectRowsParams& params, cudaStream_t stream) {
  SelectRowsParams p = params;
  if (p.n_blocks <= 0) return cudaSuccess;
  p.sel_slots = static_cast<unsigned int>(next_pow2(p.topk < 2048 ? 2048 : p.topk));
  const int smem = kFineBins * 4 + 2 * static_cast<int>(p.sel_slots) * static_cast<int>(sizeof(uint64_t));
  // many short rows: three small CTAs an SM hide one another's barriers; otherwise a row gets all the threads it can use
  if (p.row_flag != nullptr) return launch_select_rows_n<1024, true>(p, smem, stream);
  if (p.n_blocks > 2 * sm_count() && p.N <= kSelDirect) return launch_select_rows_n<512, false>(p, smem, stream);
  return launch_select_rows_n<1024, false>(p, smem, stream);
}

}  // namespace lt
