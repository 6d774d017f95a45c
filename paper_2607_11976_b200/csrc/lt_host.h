// Host-side declarations shared by the library's translation units (not part of the public ABI).
#pragma once

#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>

#include <atomic>
#include <utility>

#include "lt_common.cuh"

namespace lt {

// Lets a kernel use all the dynamic shared memory an SM has (and clusters of 16).  A property of the loaded function on a device,
// set once for each: `done` holds one bit per device and belongs to that kernel alone.
inline cudaError_t allow_smem(const void* kernel, std::atomic<unsigned long long>& done, bool wide_clusters = false) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  const unsigned long long bit = 1ull << (dev & 63);
  if (done.load(std::memory_order_acquire) & bit) return cudaSuccess;
  cudaFuncAttributes a;
  e = cudaFuncGetAttributes(&a, kernel);
  if (e != cudaSuccess) return e;
  e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024 - static_cast<int>(a.sharedSizeBytes));
  if (e == cudaSuccess && wide_clusters) e = cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  if (e == cudaSuccess) done.fetch_or(bit, std::memory_order_release);
  return e;
}

// SMs of the current device, asked for once
inline int sm_count() {
  static std::atomic<int> cached[64];
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 148;
  int n = cached[dev].load(std::memory_order_relaxed);
  if (n == 0) {
    if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n <= 0) n = 148;
    cached[dev].store(n, std::memory_order_relaxed);
  }
  return n;
}

// Clusters of `cluster` CTAs of a kernel that the current device (or the part of it that this process may use) holds at once; 0 where
// it can place none.
template <typename... Params>
inline int clusters_at_once(void (*kernel)(Params...), int threads, size_t smem, int cluster) {
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = static_cast<unsigned int>(cluster);
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(static_cast<unsigned int>(cluster));
  cfg.blockDim = dim3(static_cast<unsigned int>(threads));
  cfg.dynamicSmemBytes = smem;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  int n = 0;
  if (cudaOccupancyMaxActiveClusters(&n, kernel, &cfg) == cudaSuccess) return n;
  cudaGetLastError();
  return 0;
}
// The widest cluster of up to 16 CTAs with `smem` bytes each that the current device can place, found once for each device: cache[dev]
// belongs to that kernel.
template <typename... Params>
inline int widest_cluster(void (*kernel)(Params...), int threads, size_t smem, std::atomic<signed char>* cache) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return 1;
  int width = cache[dev & 63].load(std::memory_order_relaxed);
  if (width == 0) {
    for (width = 16; width > 1 && clusters_at_once(kernel, threads, smem, width) < 1;) width >>= 1;
    cache[dev & 63].store(static_cast<signed char>(width), std::memory_order_relaxed);
  }
  return width;
}

// Launch of a kernel that calls chain_wait (see lt_common.cuh), optionally in clusters of `cluster` CTAs.
template <typename... Params, typename... Args>
inline cudaError_t launch_chained(void (*kernel)(Params...), dim3 grid, dim3 block, size_t smem, cudaStream_t stream, int cluster,
                                  Args&&... args) {
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = static_cast<unsigned int>(cluster);
  attr[1].val.clusterDim.y = 1;
  attr[1].val.clusterDim.z = 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cfg.attrs = attr;
  cfg.numAttrs = cluster > 1 ? 2 : 1;
  return cudaLaunchKernelEx(&cfg, kernel, std::forward<Args>(args)...);
}

constexpr int kModeFilter = 0;
constexpr int kModeDump = 1;
constexpr int kRowsPerBlock = 8;     // query rows one scan CTA (and one k-NN fallback block) keeps resident
constexpr int kRowsPerBlockFp8 = 6;  // ... of the alternative fp8 scan (LT_PATH_FUSED_ABS, lt_scan_fp8.cu)
constexpr int kLinTerms = 5;         // e4m3 terms of the linear part of a query (alternative fp8 scan)
constexpr int kLinScaleStride = 8;   // floats per row of the linear-term scale table

// Parameters of the tensor-core scan kernel (lt_scan_mma.cu).
struct ScanParams {
  const float* w;          // [T][64]
  const float* k_scale;    // per key of the view, or null
  long long ks_stride;     // k_scale index of view key s is s * ks_stride
  int T;                   // rows of q / w
  int row_begin, row_end;  // rows handled by this launch (ignored when fb_list is set)
  int n_keys;              // keys in the view
  int causal_offset;       // row t sees view keys 0 .. causal_offset + t
  int skip_masked_tiles;   // 1: do not visit key tiles no row of the block can see
  int seg_tiles;           // key tiles per work item
  int topk;
  // filter mode
  float* thr;              // [T] gate: lower edge of the row's threshold bin (-inf = accept all)
  const float* smin;       // [T] sampled minimum score
  const float* width;      // [T] bin width
  unsigned int* tail;      // [T] survivors appended so far (may exceed cap)
  unsigned int* hist;      // [T][kBins]
  uint2* cand;             // [T][cap] (score bits, key index)
  int cap;
  // dump mode
  float* dump;             // dense scores
  long long dump_ld;       // row pitch of dump in floats
  // exact-fallback dump: blocks come from a device-side list, slot j of this round
  // is block fb_list[fb_round_base + j], its rows go to dump rows 8j .. 8j+7
  const int* fb_list;
  const int* fb_blocks;    // device counter: entries in fb_list
  int fb_round_base;
  int fb_slots;
  // paged key cache (null: keys are one dense matrix): logical page j of 64 keys is physical page page_table[j] of
  // the pool the key tensor map covers; k_scale is then indexed by physical row
  const int* page_table;
  int n_pages;
  long long pool_pages;    // pages of the pool behind page_table (bounds checks of the debug build)
  unsigned int wait_limit_us;  // bound of every device-side wait (0 is replaced by the default at launch)
  int debug_flags;         // LT_DEBUG_* test hooks
  // alternative fp8 scan only: the linear part of Eq. 1 prepared by launch_lin_terms
  const void* lin_q;       // [T][kLinTerms][128] e4m3 codes
  const float* lin_scale;  // [T][kLinScaleStride], the first kLinTerms entries of a row are used
  Control* ctl;
  unsigned char* status_slots;  // null: status bits are OR-ed into ctl; else ctl is cleared and every CTA leaves its bits here (lt_common.cuh)
};
constexpr int kPageKeys = 64;  // keys per page of a paged key cache

bool scan_mma_supported(int dtype, int H, int D);
// ---- lt_scan_fp8.cu: the alternative fp8 scan (|x| form of Eq. 1 with linear-term columns) ------------
// bytes of the linear-term operand rows / of the scale table of T query rows
inline size_t lin_q_bytes(int T) { return static_cast<size_t>(T) * kLinTerms * 128; }
inline size_t lin_scale_bytes(int T) { return static_cast<size_t>(T) * kLinScaleStride * 4; }
// pre-pass: q [T][64][128] e4m3, w [T][64] -> lin_q, lin_scale
cudaError_t launch_lin_terms(const void* q, const float* w, int T, void* lin_q, float* lin_scale, cudaStream_t stream);
cudaError_t launch_scan_fp8(int mode, const void* q, int T, const void* k, long long n_keys_view, long long key_pitch_elems,
                            const ScanParams& p, int grid, cudaStream_t stream);

// One warp waits, with the bounded wait every scan kernel uses, on a barrier nobody arrives at:
// result2[0] = what the wait returned (0 = gave up), result2[1] = the abort flag it left behind.
cudaError_t launch_wait_timeout_probe(unsigned int limit_us, int* result2, cudaStream_t stream);
// bare FP8 UMMA stream (measurement aid): grid CTAs, an even number when pair is set
cudaError_t launch_umma_stream(bool pair, int iters, int* status, int grid, cudaStream_t stream);

// q: [T][64][128]; k: view of n_keys_view rows whose pitch is key_pitch_elems elements.
cudaError_t launch_scan_mma(int dtype, int mode, const void* q, int T, const void* k, long long n_keys_view,
                            long long key_pitch_elems, const ScanParams& p, int grid, cudaStream_t stream);

// ---- lt_scan_knn.cu -------------------------------------------------------------------------
// Parameters of the tensor-core scan of the k-NN (inner-product) variant: bf16 queries [T][D], corpus view of
// n_keys rows, every row sees every key.
struct KnnScanParams {
  int T;                   // rows of q
  int row_begin, row_end;  // query rows handled by this launch
  int n_keys;              // corpus vectors in the view
  int D;                   // multiple of 64, at most 768
  int seg_tiles;           // corpus tiles (128 vectors) per work item
  int topk;
  // filter mode
  float* thr;              // [T] gate: lower edge of the row's threshold bin
  const float* smin;       // [T]
  const float* width;      // [T]
  unsigned int* tail;      // [T]
  unsigned int* hist;      // [T][kBins]
  uint2* cand;             // [T][cap]
  int cap;
  // dump mode
  float* dump;             // dense scores, row (t - row_begin)
  long long dump_ld;
  const unsigned int* fb_flag;  // fallback rounds: flag per block of 8 rows; the launch is a no-op if no block of its row range is flagged
  unsigned int wait_limit_us;   // bound of every device-side wait (0 is replaced by the default at launch)
  Control* ctl;
  unsigned char* status_slots;  // as in ScanParams
  int debug_flags;              // LT_DEBUG_* test hooks
};
bool scan_knn_supported(int D);
cudaError_t launch_scan_knn(int mode, const void* q, int T, const void* x, long long n_keys_view, long long key_pitch_elems,
                            const KnnScanParams& p, int grid, cudaStream_t stream);

// ---- lt_select.cu ---------------------------------------------------------------------------
// Clears `bytes` bytes at p (16-byte aligned, a multiple of 16): a kernel and not a memset, so that it chains.
cudaError_t launch_zero(void* p, size_t bytes, cudaStream_t stream);

// clear_ctl: a control block to clear on the way, or null.
// Generic SIMT scoring (any H, D, dtype): dense scores of rows [row_begin, row_end), -inf where masked.
cudaError_t launch_simt_scores(int dtype, const void* q, const float* w, const void* k, const float* k_scale, int T, int N,
                               int H, int D, int causal_offset, int row_begin, int row_end, float* out, long long ld,
                               Control* clear_ctl, cudaStream_t stream);

// Sample statistics (paper Sec. 3.2 "Sampling"): per row min / max of the sampled scores, bin
// width, and the threshold edge of the bin holding the rank-th largest sampled score.
// open (or null): what the call's later kernels want cleared; the row's CTA does it on the way.
struct OpenParams {
  Control* ctl;
  const unsigned char* status_slots;  // n_slots of them were written by the scan of the sample; 0: there was none, and ctl is cleared here
  int n_slots;
  unsigned int* tail;        // [T]
  unsigned int* hist;        // [T][kBins]
  unsigned char* row_flag;   // [T]
  unsigned int* block_flag;  // [n_blocks]
  int rows_per_block;
  int n_blocks;
};
cudaError_t launch_sample_stats(const float* sample, int T, int n_sample, int rank, float* smin, float* width, float* thr,
                                const OpenParams* open, cudaStream_t stream);

// Final selection from the candidate buffers (paper Sec. 3.2 "Top-k Selection"); rows that cannot
// be finished exactly are flagged and their block appended to the fallback list.
struct FinalSelectParams {
  const unsigned int* tail;
  const unsigned int* hist;
  const uint2* cand;
  const float* smin;
  const float* width;
  int cap, T, N, topk, causal_offset;
  int32_t* out_idx;
  float* out_score;
  unsigned char* row_flag;    // [T] 1 = needs the fallback
  unsigned int* block_flag;   // [ceil(T / rows_per_block)]
  int* fb_list;               // [ceil(T / rows_per_block)]
  int rows_per_block;         // rows of one fallback block (the scan kernel's query block)
  Control* ctl;
};
cudaError_t launch_final_select(const FinalSelectParams& p, cudaStream_t stream);

// Full-row exact select over dense scores.  Direct mode: block b handles row row_begin + b whose
// scores start at scores + b * ld.  Fallback mode (fb_list != null), R = rows_per_block: block b handles row
// fb_list[fb_round_base + b / R] * R + b % R if that row is flagged; scores at scores + b * ld.
struct SelectRowsParams {
  const float* scores;
  long long ld;
  int n_blocks;  // CTAs to launch
  int row_begin;
  int T, N, topk, causal_offset;
  int32_t* out_idx;
  float* out_score;
  const int* fb_list;
  const int* fb_blocks;
  int fb_round_base;
  int rows_per_block;
  const unsigned char* row_flag;
  Control* ctl;
  const unsigned char* status_slots;  // not null: the scan's n_slots status bytes (dense form)
  int n_slots;
  // NaN scores rank as their bit patterns do, above +inf.  nan_last != 0: they are selected only where a row has too few others,
  // which is what becomes of them in the sampled form (its gate lets none pass; a row that is then short of keys is redone)
  int nan_last;
  unsigned int sel_slots;  // set by the launch: a power of two >= topk
  int slice_keys;          // set by the launch of the cluster form
};
cudaError_t launch_select_rows(const SelectRowsParams& p, cudaStream_t stream);
// The same for few rows (direct mode only): long rows are shared by clusters of CTAs.  scores 16-byte aligned, ld a
// multiple of 4.
cudaError_t launch_select_dense(const SelectRowsParams& p, cudaStream_t stream);

// ---- lt_sampler.cu --------------------------------------------------------------------------
// counts[p] += occurrences of p in idx[0..n) (entries outside [0, N) are skipped); counts must be zeroed.
cudaError_t launch_count_positions(const int32_t* idx, long long n, int N, unsigned int* counts, cudaStream_t stream);
// the n_out most frequent positions of counts[0..N), (count desc, position asc); max_count bounds every count; scratch: rank_scratch_bytes(n_out)
size_t rank_scratch_bytes(int n_out);
cudaError_t launch_rank_counts(const unsigned int* counts, int N, int n_out, unsigned long long max_count, void* scratch,
                               int32_t* out_pos, int32_t* out_count, cudaStream_t stream);
// dense copy of the key rows (row_bytes each, multiple of 16) and scales at the sampled positions (sample_idx, or
// j * stride when it is null); page_table (or null) translates positions to physical rows of a paged key cache
// (pool_rows and ctl serve the bounds-checking build: a translated row outside the pool is read as row 0 and flagged)
cudaError_t launch_gather_keys(const void* k, const float* k_scale, const int32_t* sample_idx, long long stride, int n_sample,
                               int N, int row_bytes, const int* page_table, long long pool_rows, Control* ctl, void* out_k,
                               float* out_scale, cudaStream_t stream);

// ---- lt_dsa_union.cu ------------------------------------------------------------------------
// LiteDSA union list + membership masks of consecutive groups of `group` rows (paper Sec. 3.3).
// union_pos [n_groups][group * topk] (-1 beyond union_len), mask [T][ceil(group * topk / 32)].
cudaError_t launch_dsa_union(const int32_t* idx, int T, int topk, int N, int group, int32_t* union_pos, int32_t* union_len,
                             uint32_t* mask, cudaStream_t stream);

}  // namespace lt
