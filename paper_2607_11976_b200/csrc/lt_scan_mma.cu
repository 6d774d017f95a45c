// Tensor-core scan kernel of the fused indexer top-k (sm_100a: TMA -> shared -> tcgen05.mma -> TMEM).
//
// One CTA keeps a block of 8 query rows (8 x 64 heads = 512 operand rows of D = 128) resident in
// shared memory and streams 128-key tiles of K past it.  Per key tile it issues two 128 x 256 x 128
// UMMAs (unit u = queries 4u .. 4u+3) into the two 256-column halves of TMEM; lanes index keys and
// columns index (query, head), so each epilogue thread owns one key and finishes Eq. 1 of the paper
// (ReLU, head-weighted sum, key scale) as an in-thread chain of packed FMAs over TMEM columns.
//
//   kMode == kModeFilter  paper Sec. 3.2 "Filtering": gate the score against the row's threshold
//                         edge, ballot-compact the survivors of each warp into a staging list; a flush
//                         appends the list to the row's candidate buffer and counts its entries in the
//                         row's bin histogram; a spare warp re-derives the
//                         threshold bin from the histogram while the scan runs ("Threshold
//                         Refresh") and publishes it by plain store.
//   kMode == kModeDump    write every score (or -inf where masked) to a dense matrix: used for the
//                         sample phase, lt_indexer_scores, the unfused baseline and the exact fallback.
//
// Warp roles (608 threads): 0 TMA producer, 1 UMMA issuer (+ TMEM owner), 2 threshold refresh,
// 3..18 epilogue in four warpgroups.  Warpgroup g finishes query g of unit 0 (TMEM half 0) and then
// query g of unit 1 (half 1) of every key tile, so the UMMA warp refills one half while the other
// is drained.  A warp pulls its 64 columns of a half into registers with one wait, hands the half
// back at once and only then does the arithmetic; the four warps of a scheduler cover each
// other's barrier and TMEM latencies.  Survivors of the gate go to small
// per-warp staging lists in shared memory and are flushed to the row's candidate buffer in batches
// (one tail atomic per flush; paper Sec. 3.2 "Filtering").
#include <cuda.h>
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <type_traits>

#include "lt_common.cuh"
#include "lt_host.h"
#include "lt_ptx.cuh"
#include "lt_work_items.h"

namespace lt {

using namespace ptx;

namespace {

constexpr int kH = 64;
constexpr int kD = 128;
constexpr int kBlockQ = 8;                  // query rows resident per CTA
constexpr int kUnitQ = 4;                   // query rows per UMMA (N = 4 * 64 = 256 columns)
constexpr int kUnits = kBlockQ / kUnitQ;    // UMMAs per key tile = TMEM halves
constexpr int kTmemCols = 512;              // two accumulators of 256 fp32 columns
constexpr int kFirstEpiWarp = 3;
constexpr int kEpiWarps = 16;
constexpr int kEpiThreads = kEpiWarps * 32;
constexpr int kThreads = kFirstEpiWarp * 32 + kEpiThreads;
constexpr int kSwizzleTile = 128 * 128;     // bytes: 128 rows x 128-byte swizzled rows
constexpr int kQTile = 256 * 128;           // bytes: 256 rows x 128-byte rows (one unit, one K-half)
constexpr int kStageLen = 64;               // entries of one per-warp staging list
constexpr int kUnitWBytes = kUnitQ * kH * 4;  // bytes between the weights of query g and query 4 + g

// kU: units of four queries per key tile.  kUQ: queries a unit really has.  A chunk of more than four rows runs with
// kU = 2, kUQ = 4: unit u of every tile goes to TMEM half u, warpgroup g finishes query g of it.  A chunk of at most four
// rows (decode, verification of drafted tokens) has one unit per tile of kUQ = 1, 2 or 4 queries: its UMMAs are 64 kUQ
// columns wide, the TMEM holds 512 / (64 kUQ) accumulators that consecutive tiles rotate through, and the four
// warpgroups take 4 / kUQ tiles at a time (warpgroup g: query g % kUQ of the tiles whose number is g / kUQ modulo
// 4 / kUQ).  One accumulator that is issued, drained and issued again (as it was) leaves both the tensor pipe and the
// epilogue waiting for the other: 1 / 4 rows over 2^20 fp8 keys 63 / 69 us; now 34 / 56 us, with 21 us the time of
// reading the keys.
template <bool kFp8, int kU, int kUQ>
struct Cfg {
  static_assert((kU == 2 && kUQ == 4) || (kU == 1 && (kUQ == 1 || kUQ == 2 || kUQ == 4)), "see above");
  static constexpr int kHalves = kFp8 ? 1 : 2;           // 128-byte row pieces along D
  static constexpr int kElemsPerRow128 = kFp8 ? 128 : 64;  // elements in a 128-byte row
  static constexpr int kStages = kU == 2 ? (kFp8 ? 6 : 2) : (kFp8 ? 8 : 4);  // K-tile ring depth: what the query block leaves
  static constexpr int kKBlocks = kFp8 ? 4 : 8;          // UMMA K-steps per tile (K = 32 fp8 / 16 bf16 = 32 bytes)
  static constexpr int kN = kUQ * kH;                    // UMMA columns of a unit
  static constexpr int kAccs = kTmemCols / kN;           // accumulators in TMEM
  static constexpr int kShare = kUnitQ / kUQ;            // tiles the four warpgroups work on together
  static constexpr int kDrainers = 4 * kUQ;              // warps that read one accumulator
  static constexpr int kQBytes = kU * kHalves * kQTile;
  static constexpr int kStageBytes = kHalves * kSwizzleTile;
  static constexpr int kSmemTiles = kQBytes + kStages * kStageBytes;
};

struct SmemTail {
  float w[kBlockQ * kH];
  float thr[kBlockQ];
  float smin[kBlockQ];
  float width[kBlockQ];
  float inv_width[kBlockQ];
  int vis[kBlockQ];
  int dump_row[kBlockQ];
  uint64_t bar_full[8];
  uint64_t bar_empty[8];
  uint64_t bar_q_full;
  uint64_t bar_q_empty;
  uint64_t bar_tmem_full[8];
  uint64_t bar_tmem_empty[8];
  uint32_t tmem_base;
  int abort_flag;     // [0] raised by a wait that ran out; every role unwinds on it
  int wait_limit_us;  // [1] bound of every wait (read by mbar_wait through the flag's address)
  int epi_abort;
  int done_seq;
  uint2 stage[kEpiWarps][kUnits][kStageLen];  // per warp and unit: (score bits, key index) of survivors
};

template <bool kFp8, int kU, int kUQ>
constexpr int smem_bytes() {
  return 1024 + Cfg<kFp8, kU, kUQ>::kSmemTiles + static_cast<int>(sizeof(SmemTail));
}

struct Item {
  int t0;        // first query row of the block
  int tile_lo;   // key tiles [tile_lo, tile_hi)
  int tile_hi;
  int slot;      // dump slot (fallback mode) or block number
};

// Work items are (key segment, query block) pairs, segment-major, so that CTAs running side by
// side stream the same part of K (L2 reuse) for different query blocks.  Within a segment the last rows come first: under a triangular
// mask they are the longest.  Dealt out to and fro, 4096 rows over their own 4096 keys, scan 117 -> 107 us (lt_work_items.h).
// (false also for numbers past the last item: nothing of the chunk is looked up for them)
__device__ __forceinline__ bool resolve_item(const ScanParams& p, int n_blocks, unsigned int n_items, unsigned int item, Item& it) {
  int qb;
  if (!split_item(item, n_items, n_blocks, p.seg_tiles, qb, it.tile_lo)) return false;
  int last_row;
  if (p.fb_list != nullptr) {
    it.t0 = p.fb_list[p.fb_round_base + qb] * kBlockQ;
    it.slot = qb;
    last_row = min(it.t0 + kBlockQ, p.T) - 1;
  } else {
    it.t0 = p.row_begin + qb * kBlockQ;
    it.slot = qb;
    last_row = min(it.t0 + kBlockQ, p.row_end) - 1;
  }
  int n_tiles = (p.n_keys + kTileKeys - 1) / kTileKeys;
  if (p.skip_masked_tiles) {
    int vis = visible_keys(last_row, p.n_keys, p.causal_offset);
    n_tiles = (vis + kTileKeys - 1) / kTileKeys;
  }
  it.tile_hi = min(it.tile_lo + p.seg_tiles, n_tiles);
  return it.tile_lo < it.tile_hi;
}

// Where the scale of view key s lives: at s * ks_stride, or with a paged key cache at the key's physical row.
template <bool kPaged, bool kDense = false>
__device__ __forceinline__ size_t scale_index(const ScanParams& p, int s) {
  if (kPaged) {
    long long phys = __ldg(p.page_table + (s / kPageKeys));
    if (!LT_IN_BOUNDS(phys >= 0 && phys < p.pool_pages, p.ctl)) phys = 0;  // a page-table entry outside the pool
    return static_cast<size_t>(phys) * kPageKeys + static_cast<size_t>(s % kPageKeys);
  }
  return kDense ? static_cast<size_t>(s) : static_cast<size_t>(s) * p.ks_stride;  // (the fused scan reads every key)
}

// ---- Eq. 1 for one key against one query ------------------------------------------------------
// 32 TMEM columns (per-head dots) -> ReLU -> weighted sum, accumulated into four packed fp32 pairs
// (eight independent chains).  Head h lands in pair (h / 2) % 4, lane h % 2; combine() fixes the
// order of the final additions.  These functions produce every score the library ranks or dumps
// on the tensor-core path, so fused, dumped and fallback scores agree bit for bit.
struct Acc8 {
  uint64_t p[4];
};
__device__ __forceinline__ void unpack2(uint64_t v, float& lo, float& hi) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
// acc (+)= w * ReLU(x) for two heads at once.  The ReLU is applied in place on the two registers
// the TMEM load filled, so that they stay an aligned register pair for the packed FMA.
//   kSat == false: ReLU(x) = max(x, 0)                                  (ALU pipe)
//   kSat == true : ReLU(x) = sat(x * 2^-25) * 2^25, the 2^25 being folded into the weight the
//                  caller stored for this head                          (FMA pipe)
// The saturating form needs |x| < 2^25 and no underflow of x * 2^-25; both hold for dot products of
// 128 e4m3 codes (|x| <= 448^2 * 128 < 2^25, non-zero |x| >= 2^-18).  Scaling by a power of two is
// exact, so w * 2^25 * (x * 2^-25) and w * x round to the same fp32 value: the two forms give
// bit-identical sums and are mixed only to spread the work over both pipes.
// kFirst: the accumulator starts at w * ReLU(x) (a multiply) instead of being zero-initialised.
template <bool kSat, bool kFirst>
__device__ __forceinline__ void relu_fma2(uint64_t& acc, uint64_t w, uint32_t& x0, uint32_t& x1) {
  // everything stays in the untyped 32-bit registers of the TMEM load (no typed copies)
  if (kSat) {
    asm("mul.sat.f32 %0, %0, 0f33000000;" : "+r"(x0));
    asm("mul.sat.f32 %0, %0, 0f33000000;" : "+r"(x1));
  } else {
    asm("max.f32 %0, %0, 0f00000000;" : "+r"(x0));
    asm("max.f32 %0, %0, 0f00000000;" : "+r"(x1));
  }
  if (kFirst) {
    asm("{\n.reg .b64 x;\nmov.b64 x, {%1, %2};\nmul.rn.f32x2 %0, %3, x;\n}\n" : "=l"(acc) : "r"(x0), "r"(x1), "l"(w));
  } else {
    asm("{\n.reg .b64 x;\nmov.b64 x, {%1, %2};\nfma.rn.f32x2 %0, %3, x, %0;\n}\n" : "+l"(acc) : "r"(x0), "r"(x1), "l"(w));
  }
}
// Weight stored in shared memory for head h: heads whose ReLU takes the saturating form carry 2^25.
template <bool kFp8>
__device__ __forceinline__ float stored_weight(float w, int h) {
  return (kFp8 && (h & 2)) ? w * 33554432.f : w;
}
// Eight heads starting at column J of a 32-column piece.  kOff: byte offset of the piece's weights
// from w_addr, folded into the load instructions as an immediate.
template <bool kFp8, bool kFirst, int kOff, int J>
__device__ __forceinline__ void head_sum8(uint32_t (&v)[32], uint32_t w_addr, Acc8& acc) {
  uint64_t w01, w23, w45, w67;
  asm volatile("ld.shared.v2.b64 {%0, %1}, [%2+%3];" : "=l"(w01), "=l"(w23) : "r"(w_addr), "n"(kOff + J * 4));
  asm volatile("ld.shared.v2.b64 {%0, %1}, [%2+%3];" : "=l"(w45), "=l"(w67) : "r"(w_addr), "n"(kOff + J * 4 + 16));
  constexpr bool first = kFirst && J == 0;
  relu_fma2<false, first>(acc.p[0], w01, v[J + 0], v[J + 1]);
  relu_fma2<kFp8, first>(acc.p[1], w23, v[J + 2], v[J + 3]);
  relu_fma2<false, first>(acc.p[2], w45, v[J + 4], v[J + 5]);
  relu_fma2<kFp8, first>(acc.p[3], w67, v[J + 6], v[J + 7]);
}
template <bool kFp8, bool kFirst, int kOff>
__device__ __forceinline__ void head_sum32(uint32_t (&v)[32], uint32_t w_addr, Acc8& acc) {
  head_sum8<kFp8, kFirst, kOff, 0>(v, w_addr, acc);
  head_sum8<kFp8, kFirst, kOff, 8>(v, w_addr, acc);
  head_sum8<kFp8, kFirst, kOff, 16>(v, w_addr, acc);
  head_sum8<kFp8, kFirst, kOff, 24>(v, w_addr, acc);
}
__device__ __forceinline__ float combine(const Acc8& acc, float ks) {
  uint64_t ab, cd, all;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(ab) : "l"(acc.p[0]), "l"(acc.p[1]));
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(cd) : "l"(acc.p[2]), "l"(acc.p[3]));
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(all) : "l"(ab), "l"(cd));
  float lo, hi;
  unpack2(all, lo, hi);
  return __fmaf_rn(lo + hi, ks, 0.f);  // the + 0 turns -0 into +0
}

// Flush one staging list: reserve room in the row's candidate buffer with a single atomic, copy the
// entries out with all lanes and count each of them in the row's histogram (fire-and-forget
// atomics).  Doing the bin arithmetic here, 32 entries at a time, keeps it out of the per-tile path;
// the refresh warp merely sees the counts a little later, which can only leave the gate looser.
// Entries beyond the capacity are dropped but still counted, and the tail counter runs past the
// capacity, which is how the final select learns that the row overflowed.
// What a flush costs is its length: the accumulator half this warp reads next waits for it, and with it the UMMA and the other
// fifteen warps.  So a lane's two entries are worked on side by side, and while the reservation is under way (4096 rows over 64 K bf16
// keys, scan 3.01 -> 2.85 ms, 8192 over 128 K fp8 keys 9.76 -> 9.56, against one entry after the other behind the reservation; with the
// histogram in shared memory instead, nothing gained; out of line + 4 %).
__device__ __forceinline__ void flush_stage(const uint2* list, int count, const ScanParams& p, int t, int lane, float smin,
                                            float width, float inv_width) {
  static_assert(kStageLen == 64, "two entries per lane");
  __syncwarp();
  uint32_t base = 0;
  if (lane == 0) base = atomicAdd(p.tail + t, static_cast<uint32_t>(count));
  const bool has0 = lane < count, has1 = lane + 32 < count;
  const uint2 e0 = list[lane], e1 = list[lane + 32];  // (past the count: an older entry, not used)
  unsigned int* hist = p.hist + static_cast<size_t>(t) * kBins;
  int b0, b1;
  bins_of2(__uint_as_float(e0.x), __uint_as_float(e1.x), smin, width, inv_width, b0, b1);
  if (has0 && LT_IN_BOUNDS(b0 >= 0 && b0 < kBins && t >= 0 && t < p.T, p.ctl)) atomicAdd(hist + b0, 1u);
  if (has1 && LT_IN_BOUNDS(b1 >= 0 && b1 < kBins && t >= 0 && t < p.T, p.ctl)) atomicAdd(hist + b1, 1u);
  uint2* cand = p.cand + static_cast<size_t>(t) * p.cap;
  base = __shfl_sync(0xffffffffu, base, 0);
  const uint32_t pos0 = base + lane, pos1 = pos0 + 32u, cap = static_cast<uint32_t>(p.cap);
  if (has0 && pos0 < cap && LT_IN_BOUNDS(t >= 0 && t < p.T && e0.y < static_cast<uint32_t>(p.n_keys), p.ctl)) cand[pos0] = e0;
  if (has1 && pos1 < cap && LT_IN_BOUNDS(t >= 0 && t < p.T && e1.y < static_cast<uint32_t>(p.n_keys), p.ctl)) cand[pos1] = e1;
  __syncwarp();
}

template <bool kFp8, int kMode, bool kPaged, int kU = kUnits, int kUQ = kUnitQ>
__global__ void __launch_bounds__(kThreads, 1)
scan_kernel(const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_k, const ScanParams p) {
  using C = Cfg<kFp8, kU, kUQ>;
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw_addr = smem_u32(smem_raw);
  const uint32_t pad = (1024u - (raw_addr & 1023u)) & 1023u;
  uint8_t* smem = smem_raw + pad;
  const uint32_t q_base = raw_addr + pad;
  const uint32_t k_base = q_base + C::kQBytes;
  SmemTail* st = reinterpret_cast<SmemTail*>(smem + C::kSmemTiles);

  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;

  // a fallback round with no flagged block left has nothing to do (uniform across the CTA)
  if (p.fb_list != nullptr) {
    chain_wait();
    chain_trigger();
    if (*p.fb_blocks <= p.fb_round_base) return;
  }

  if (threadIdx.x == 0) {
    for (int i = 0; i < C::kStages; ++i) {
      mbar_init(smem_u32(&st->bar_full[i]), 1);
      mbar_init(smem_u32(&st->bar_empty[i]), 1);
    }
    mbar_init(smem_u32(&st->bar_q_full), 1);
    mbar_init(smem_u32(&st->bar_q_empty), 1);
    for (int i = 0; i < C::kAccs; ++i) {
      mbar_init(smem_u32(&st->bar_tmem_full[i]), 1);
      mbar_init(smem_u32(&st->bar_tmem_empty[i]), C::kDrainers);
    }
    st->abort_flag = 0;
    st->wait_limit_us = static_cast<int>(p.wait_limit_us);
    st->epi_abort = 0;
    st->done_seq = 0;
    fence_mbar_init();
    prefetch_tensormap(&tm_q);
    prefetch_tensormap(&tm_k);
  }
  if (warp == 1) {
    tmem_alloc(smem_u32(&st->tmem_base), kTmemCols);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = st->tmem_base;
  volatile int* abort_flag = &st->abort_flag;
  chain_wait();  // barriers, TMEM and tensor maps are ready by now
  if (kMode == kModeDump && p.status_slots != nullptr) {
    if (blockIdx.x == 0) clear_control(p.ctl, threadIdx.x);
    if (threadIdx.x == 0) store_status_slot(p.status_slots, p.ctl, 0);
  }

  // number of query blocks / items of this launch
  int n_blocks;
  if (p.fb_list != nullptr) {
    int avail = *p.fb_blocks - p.fb_round_base;
    n_blocks = avail < 0 ? 0 : (avail > p.fb_slots ? p.fb_slots : avail);
  } else {
    n_blocks = (p.row_end - p.row_begin + kBlockQ - 1) / kBlockQ;
  }
  const unsigned int n_items = count_items((p.n_keys + kTileKeys - 1) / kTileKeys, p.seg_tiles, n_blocks);
  const unsigned int n_rounds = count_rounds(n_items, gridDim.x);

  if (warp == 0) {
    // ------------------------------------------------------------------ TMA producer
    if (lane == 0) {
      int stage = 0;
      uint32_t phase = 0;
      uint32_t n_done = 0;  // items issued so far (parity of the Q-block handshake)
      bool ok = true;
      for (unsigned int round = 0; round < n_rounds && ok; ++round) {
        Item it;
        if (!resolve_item(p, n_blocks, n_items, item_of_round(round, blockIdx.x, gridDim.x), it)) continue;
        // query block: wait until the UMMAs of the previous item no longer read it
        ok = mbar_wait<40>(smem_u32(&st->bar_q_empty), (n_done & 1) ^ 1, abort_flag);
        if (!ok) break;
        mbar_arrive_expect_tx(smem_u32(&st->bar_q_full), kU * C::kHalves * kQTile);
        for (int u = 0; u < kU; ++u)
          for (int hf = 0; hf < C::kHalves; ++hf)
            tma_load_2d(q_base + (u * C::kHalves + hf) * kQTile, &tm_q, hf * C::kElemsPerRow128,
                        (it.t0 + u * kUnitQ) * kH, smem_u32(&st->bar_q_full));
        ++n_done;
        for (int tile = it.tile_lo; tile < it.tile_hi; ++tile) {
          ok = mbar_wait<40>(smem_u32(&st->bar_empty[stage]), phase ^ 1, abort_flag);
          if (!ok) break;
          // test hook (lt_tunables.debug_flags): CTA 0 never loads the first key tile of its first item, so
          // the UMMA warp's wait for it runs out and the whole CTA unwinds through the timeout path
          if ((p.debug_flags & LT_DEBUG_SKIP_ONE_KTILE) && blockIdx.x == 0 && n_done == 1 && tile == it.tile_lo) {
            ok = false;
            break;
          }
          mbar_arrive_expect_tx(smem_u32(&st->bar_full[stage]), C::kStageBytes);
          if (!kPaged) {
            for (int hf = 0; hf < C::kHalves; ++hf)
              tma_load_2d(k_base + stage * C::kStageBytes + hf * kSwizzleTile, &tm_k, hf * C::kElemsPerRow128,
                          tile * kTileKeys, smem_u32(&st->bar_full[stage]));
          } else {
            // paged key cache: a tile is two pages of 64 keys, each wherever the page table says (the map's
            // box is then 64 rows); pages past the end of the table are read from page 0 and masked later
            for (int pg = 0; pg < kTileKeys / kPageKeys; ++pg) {
              const int lp = tile * (kTileKeys / kPageKeys) + pg;
              int phys = lp < p.n_pages ? __ldg(p.page_table + lp) : 0;
              if (!LT_IN_BOUNDS(phys >= 0 && phys < p.pool_pages, p.ctl)) phys = 0;  // entry outside the pool
              for (int hf = 0; hf < C::kHalves; ++hf)
                tma_load_2d(k_base + stage * C::kStageBytes + hf * kSwizzleTile + pg * kPageKeys * 128, &tm_k,
                            hf * C::kElemsPerRow128, phys * kPageKeys, smem_u32(&st->bar_full[stage]));
            }
          }
          if (++stage == C::kStages) {
            stage = 0;
            phase ^= 1;
          }
        }
      }
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------------ UMMA issuer
    if (lane == 0) {
      constexpr uint32_t idesc = make_idesc(kFp8, C::kN);
      int stage = 0;
      uint32_t phase = 0;
      uint32_t acc_phase = 0;  // two units: flips once per key tile, each TMEM half is filled once per tile
      uint32_t useq = 0;       // one unit: tiles issued so far
      uint32_t n_done = 0;
      bool ok = true;
      for (unsigned int round = 0; round < n_rounds && ok; ++round) {
        Item it;
        if (!resolve_item(p, n_blocks, n_items, item_of_round(round, blockIdx.x, gridDim.x), it)) continue;
        ok = mbar_wait<40>(smem_u32(&st->bar_q_full), n_done & 1, abort_flag);
        if (!ok) break;
        ++n_done;
        for (int tile = it.tile_lo; tile < it.tile_hi && ok; ++tile) {
          ok = mbar_wait<40>(smem_u32(&st->bar_full[stage]), phase, abort_flag);
          if (!ok) break;
          for (int u = 0; u < kU; ++u) {
            const uint32_t acc = kU == 2 ? static_cast<uint32_t>(u) : useq % C::kAccs;
            const uint32_t par = kU == 2 ? acc_phase ^ 1 : ((useq / C::kAccs) & 1) ^ 1;
            ok = mbar_wait<40>(smem_u32(&st->bar_tmem_empty[acc]), par, abort_flag);
            if (!ok) break;
            tc_fence_after();
#pragma unroll
            for (int kb = 0; kb < C::kKBlocks; ++kb) {
              const int hf = kFp8 ? 0 : (kb >> 2);
              const int step = kFp8 ? kb : (kb & 3);
              uint64_t a = make_smem_desc_sw128(k_base + stage * C::kStageBytes + hf * kSwizzleTile) + (step * 32 >> 4);
              uint64_t b = make_smem_desc_sw128(q_base + (u * C::kHalves + hf) * kQTile) + (step * 32 >> 4);
              tc_mma<kFp8>(tmem_base + acc * C::kN, a, b, idesc, kb > 0 ? 1u : 0u);
            }
            tc_commit(smem_u32(&st->bar_tmem_full[acc]));
          }
          acc_phase ^= 1;
          ++useq;
          tc_commit(smem_u32(&st->bar_empty[stage]));
          if (++stage == C::kStages) {
            stage = 0;
            phase ^= 1;
          }
        }
        tc_commit(smem_u32(&st->bar_q_empty));
      }
    }
  } else {
    // ------------------------------------------------------------------ epilogue (+ refresh warp)
    const bool is_refresh = (warp == 2);
    const int n_sync = (kMode == kModeFilter) ? kEpiThreads + 32 : kEpiThreads;
    if (!(is_refresh && kMode != kModeFilter)) {
      const int e = threadIdx.x - kFirstEpiWarp * 32;  // epilogue thread number (valid for epilogue warps)
      const int ew = warp - kFirstEpiWarp;             // epilogue warp number
      const int quarter = warp & 3;                    // TMEM lane quarter this warp may read
      const int g = (ew >> 2) % kUQ;                   // warpgroup 0..3: queries g (unit 0) and 4 + g (unit 1)
      const uint32_t turn = static_cast<uint32_t>((ew >> 2) / kUQ);  // one unit: which of kShare consecutive tiles it takes
      const int key_in_tile = quarter * 32 + lane;
      const uint32_t tcol = tmem_base + (static_cast<uint32_t>(quarter * 32) << 16) + static_cast<uint32_t>(g * kH);
      const uint32_t w_addr = smem_u32(st->w) + g * kH * 4;
      uint32_t acc_phase = 0;
      uint32_t useq = 0;  // one unit: tiles gone through so far
      int seq = 0;
      for (unsigned int round = 0; round < n_rounds; ++round) {
        Item it;
        if (!resolve_item(p, n_blocks, n_items, item_of_round(round, blockIdx.x, gridDim.x), it)) continue;
        ++seq;
        named_bar_sync(1, n_sync);  // A: everybody is done with the previous item's shared state
        if (!is_refresh) {
          for (int i = e; i < kBlockQ * kH; i += kEpiThreads) {
            int t = it.t0 + i / kH;
            st->w[i] = (t < p.T) ? stored_weight<kFp8>(p.w[static_cast<size_t>(t) * kH + (i % kH)], i % kH) : 0.f;
          }
          if (e < kBlockQ) {
            int t = it.t0 + e;
            bool live = (p.fb_list != nullptr) ? (t < p.T) : (t < p.row_end);
            st->vis[e] = live ? visible_keys(t, p.n_keys, p.causal_offset) : 0;
            st->dump_row[e] = live ? ((p.fb_list != nullptr) ? it.slot * kBlockQ + e : t - p.row_begin) : -1;
            if (kMode == kModeFilter) {
              st->thr[e] = live ? __ldcg(p.thr + t) : INFINITY;
              st->smin[e] = live ? p.smin[t] : 0.f;
              st->width[e] = live ? p.width[t] : 0.f;
              st->inv_width[e] = (live && p.width[t] > 0.f) ? 1.f / p.width[t] : 0.f;
            }
          }
          if (e == 0) st->epi_abort = *abort_flag;
        }
        named_bar_sync(1, n_sync);  // B: shared state of this item is ready
        if (st->epi_abort) break;

        if (is_refresh) {
          // ---- paper Sec. 3.2 "Threshold Refresh": walk each row's histogram from the top bin
          // down until the cumulative count reaches k; publish the bin's lower edge by plain store.
          // The gate moves fast only while few keys have been seen, so the polling interval grows
          // geometrically (1 us -> 32 us): a stale edge merely admits a few more candidates, while a
          // busy polling warp would take issue slots from the epilogue warps of its scheduler.
          int cur_tb[kBlockQ];
#pragma unroll
          for (int r = 0; r < kBlockQ; ++r) cur_tb[r] = 0;
          unsigned int sleep_ns = 1000;
          while (true) {
#pragma unroll
            for (int r = 0; r < kBlockQ; ++r) {
              int t = it.t0 + r;
              if (t >= p.row_end) continue;
              const uint4* hp = reinterpret_cast<const uint4*>(p.hist + static_cast<size_t>(t) * kBins + lane * 8);
              uint4 h0 = __ldcg(hp), h1 = __ldcg(hp + 1);
              uint32_t c[8] = {h0.x, h0.y, h0.z, h0.w, h1.x, h1.y, h1.z, h1.w};
              uint32_t mine = c[0] + c[1] + c[2] + c[3] + c[4] + c[5] + c[6] + c[7];
              // suffix sum over lanes: above = total count in bins owned by higher lanes
              uint32_t incl = mine;
#pragma unroll
              for (int d = 1; d < 32; d <<= 1) {
                uint32_t o = __shfl_down_sync(0xffffffffu, incl, d);
                if (lane + d < 32) incl += o;
              }
              uint32_t above = incl - mine;
              bool crosses = (above < static_cast<uint32_t>(p.topk)) && (incl >= static_cast<uint32_t>(p.topk));
              uint32_t who = __ballot_sync(0xffffffffu, crosses);
              if (who) {
                int src = __ffs(who) - 1;  // exactly one lane crosses
                int tb = 0;
                if (lane == src) {
                  uint32_t cum = above;
                  for (int j = 7; j >= 0; --j) {
                    cum += c[j];
                    if (cum >= static_cast<uint32_t>(p.topk)) {
                      tb = lane * 8 + j;
                      break;
                    }
                  }
                }
                tb = __shfl_sync(0xffffffffu, tb, src);
                if (tb > cur_tb[r]) {
                  cur_tb[r] = tb;
                  if (lane == 0) {
                    float edge = bin_edge(tb, st->smin[r], st->width[r]);
                    // never lower the gate this CTA already uses (the sample's edge may be higher)
                    if (edge > *reinterpret_cast<volatile float*>(&st->thr[r])) {
                      *reinterpret_cast<volatile float*>(&st->thr[r]) = edge;
                      __stcg(p.thr + t, edge);
                    }
                  }
                }
              }
            }
            // sleep in slices so that the end of the item is noticed quickly; lane 0 reads the flags and the
            // whole warp follows its decision, so that no lane can leave while others still execute the
            // full-mask shuffles above
            bool done = false;
            for (unsigned int slept = 0; slept < sleep_ns && !done; slept += 1000) {
              __nanosleep(1000);
              int d = 0;
              if (lane == 0) d = (*reinterpret_cast<volatile int*>(&st->done_seq) >= seq || *abort_flag) ? 1 : 0;
              done = __shfl_sync(0xffffffffu, d, 0) != 0;
            }
            if (done) break;
            if (sleep_ns < 32000) sleep_ns += sleep_ns >> 1;
          }
          continue;
        }

        // ---- epilogue proper: this warp finishes queries g and 4 + g for its 32 keys of every tile.  The loop is bound by
        // instruction issue, so what is not arithmetic is kept out of it: tiles that every row sees whole have a loop of their own
        // without the visibility test, the key scale's address is clamped instead of tested, waits poll out of line and
        // failures are looked at once per tile (512 rows over 2^20 fp8 keys 5.10 -> 4.84 ms, 4096 over 128 K 5.42 -> 5.17, bf16
        // over 64 K 3.55 -> 3.43).
        // Every step with a long fixed latency is issued ahead of its use: the key scale of the
        // next tile and the row threshold are fetched before the arithmetic of the current one.
        int cnt[kUnits] = {0, 0};  // entries in this warp's staging lists (warp-uniform)
        const int vis_first = st->vis[0];
        const bool has_scale = p.k_scale != nullptr;
        bool ok = true;
        float ks_next = 1.f;
        // with one unit per tile, the first tile of the item that is this warpgroup's turn
        const int tile_first = kU == 2 ? it.tile_lo : it.tile_lo + static_cast<int>((turn - useq) % C::kShare);
        // (clamped instead of skipped past the last key: a load nobody uses is cheaper than the tests)
        auto fetch_scale = [&](int s) {
          if (kFp8 || has_scale) ks_next = __ldg(p.k_scale + scale_index<kPaged, kMode == kModeFilter>(p, min(s, p.n_keys - 1)));
        };
        fetch_scale(tile_first * kTileKeys + key_in_tile);
        int tile = tile_first;
        // kPartial: some row of the block may not see some key of the tile (diagonal or ragged last tile)
        auto run_tiles = [&](int tile_end, auto partial_tag) {
          constexpr bool kPartial = decltype(partial_tag)::value;
          for (; tile < tile_end && ok; tile += C::kShare) {
            const int s = tile * kTileKeys + key_in_tile;
            const float ks = ks_next;
            fetch_scale(s + C::kShare * kTileKeys);
#pragma unroll
            for (int u = 0; u < kU; ++u) {
              const int r = u * kUnitQ + g;
              float thr = 0.f;
              if (kMode == kModeFilter) thr = *reinterpret_cast<volatile float*>(&st->thr[r]);
              const uint32_t tseq = useq + static_cast<uint32_t>(tile - it.tile_lo);
              const uint32_t ab = kU == 2 ? static_cast<uint32_t>(u) : tseq % C::kAccs;
              // (a failed wait is acted on at the end of the tile: until then values nobody uses go through the motions)
              if (!mbar_wait_hot(smem_u32(&st->bar_tmem_full[ab]), kU == 2 ? acc_phase : (tseq / C::kAccs) & 1, abort_flag)) ok = false;
              tc_fence_after();
              // the 64 columns of this query: both loads in flight, one wait.  The loads are issued even
              // after a failed wait (they then fetch values nobody uses): keeping them unconditional
              // keeps the 64 destination registers free of copies.
              uint32_t va[32], vb[32];
              tmem_ld32(tcol + ab * C::kN, va);
              tmem_ld32(tcol + ab * C::kN + 32, vb);
              tmem_ld_wait();
              // this warp's columns of half u are in registers: hand the half back to the UMMA warp
              tc_fence_before();
              __syncwarp();
              if (lane == 0) mbar_arrive(smem_u32(&st->bar_tmem_empty[ab]));
              Acc8 acc;
              if (u == 0) {
                head_sum32<kFp8, true, 0>(va, w_addr, acc);
                head_sum32<kFp8, false, 128>(vb, w_addr, acc);
              } else {
                head_sum32<kFp8, true, kUnitWBytes>(va, w_addr, acc);
                head_sum32<kFp8, false, kUnitWBytes + 128>(vb, w_addr, acc);
              }
              const float score = combine(acc, ks);
              if (kMode == kModeDump) {
                const int dr = st->dump_row[r];
                if (dr >= 0 && s < p.n_keys &&
                    LT_IN_BOUNDS(s < p.dump_ld && dr < (p.fb_list != nullptr ? p.fb_slots * kBlockQ : p.row_end - p.row_begin), p.ctl))
                  p.dump[static_cast<size_t>(dr) * p.dump_ld + s] = (s < st->vis[r]) ? score : -INFINITY;
              } else {
                // ---- paper Sec. 3.2 "Filtering": gate, ballot-compact into the warp's staging list,
                // count in the histogram; the list is flushed to the candidate buffer in batches
                bool pass = score >= thr;
                if (kPartial) pass = pass && (s < st->vis[r]);
                const uint32_t ballot = __ballot_sync(0xffffffffu, pass);
                if (ballot != 0) {
                  const int t = it.t0 + r;
                  const int n = __popc(ballot);
                  uint2* list = st->stage[ew][u];
                  if (cnt[u] + n > kStageLen) {
                    flush_stage(list, cnt[u], p, t, lane, st->smin[r], st->width[r], st->inv_width[r]);
                    cnt[u] = 0;
                  }
                  if (pass) list[cnt[u] + __popc(ballot & ((1u << lane) - 1u))] = make_uint2(__float_as_uint(score), static_cast<uint32_t>(s));
                  cnt[u] += n;
                }
              }
            }
            acc_phase ^= 1;
          }
        };
        if (kMode == kModeFilter) run_tiles(min(it.tile_hi, vis_first / kTileKeys), std::false_type{});
        run_tiles(it.tile_hi, std::true_type{});
        useq += static_cast<uint32_t>(it.tile_hi - it.tile_lo);
        if (kMode == kModeFilter) {
#pragma unroll
          for (int u = 0; u < kU; ++u)
            if (cnt[u] > 0) {
              const int r = u * kUnitQ + g;
              flush_stage(st->stage[ew][u], cnt[u], p, it.t0 + r, lane, st->smin[r], st->width[r], st->inv_width[r]);
            }
        }
        if (warp == kFirstEpiWarp && lane == 0) *reinterpret_cast<volatile int*>(&st->done_seq) = seq;
      }
    }
  }

  // ---------------------------------------------------------------------- teardown
  __syncwarp();
  tc_fence_before();
  __syncthreads();
  if (st->abort_flag) {
    if (threadIdx.x == 0) {
      if (p.status_slots != nullptr) {
        store_status_slot(p.status_slots, p.ctl, LT_STATUS_TIMEOUT);
      } else {
        atomicOr(&p.ctl->status, LT_STATUS_TIMEOUT);
      }
    }
    // give copies and UMMAs still in flight time to land before TMEM and shared memory go away
    uint64_t t0 = globaltimer_ns();
    while (globaltimer_ns() - t0 < 200000ull) __nanosleep(1000);
    __syncthreads();
  }
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem_base, kTmemCols);
  }
}

// ---------------------------------------------------------------------------------------------
// host side: tensor maps and launch
// ---------------------------------------------------------------------------------------------
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                                  const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn get_encode_fn() {
  static EncodeTiledFn fn = nullptr;
  if (fn == nullptr) {
    void* ptr = nullptr;
    cudaDriverEntryPointQueryResult qres;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &ptr, cudaEnableDefault, &qres) != cudaSuccess ||
        qres != cudaDriverEntryPointSuccess)
      return nullptr;
    fn = reinterpret_cast<EncodeTiledFn>(ptr);
  }
  return fn;
}

// 2-D map over a row-major [rows][kD] matrix with a given row pitch; box = 128 bytes x box_rows,
// 128-byte swizzle, zero fill outside the matrix.
bool make_map(CUtensorMap* map, bool fp8, const void* base, uint64_t rows, uint64_t pitch_bytes, uint32_t box_rows) {
  EncodeTiledFn enc = get_encode_fn();
  if (enc == nullptr) return false;
  cuuint64_t dims[2] = {static_cast<cuuint64_t>(kD), rows};
  cuuint64_t strides[1] = {pitch_bytes};
  cuuint32_t box[2] = {static_cast<cuuint32_t>(fp8 ? 128 : 64), box_rows};
  cuuint32_t estr[2] = {1, 1};
  CUresult r = enc(map, fp8 ? CU_TENSOR_MAP_DATA_TYPE_UINT8 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base),
                   dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                   CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS;
}

template <bool kFp8, int kMode, bool kPaged, int kU, int kUQ>
cudaError_t launch_one(const CUtensorMap& tq, const CUtensorMap& tk, const ScanParams& p, int grid, cudaStream_t stream) {
  constexpr int bytes = smem_bytes<kFp8, kU, kUQ>();
  static std::atomic<unsigned long long> done{0};
  cudaError_t e = allow_smem(reinterpret_cast<const void*>(scan_kernel<kFp8, kMode, kPaged, kU, kUQ>), done);
  if (e != cudaSuccess) return e;
  return launch_chained(scan_kernel<kFp8, kMode, kPaged, kU, kUQ>, grid, kThreads, bytes, stream, 1, tq, tk, p);
}
// the paged variant is a separate instantiation so that the dense kernels carry none of its address arithmetic; the
// one-unit variants serve chunks of at most kUnitQ rows (see Cfg)
template <bool kFp8, int kMode, bool kPaged>
cudaError_t launch_paged(const CUtensorMap& tq, const CUtensorMap& tk, const ScanParams& p, int grid, cudaStream_t stream) {
  const int rows = p.fb_list == nullptr ? p.row_end - p.row_begin : kBlockQ;
  if (rows > kUnitQ) return launch_one<kFp8, kMode, kPaged, kUnits, kUnitQ>(tq, tk, p, grid, stream);
  if (rows > 2) return launch_one<kFp8, kMode, kPaged, 1, 4>(tq, tk, p, grid, stream);
  if (rows == 2) return launch_one<kFp8, kMode, kPaged, 1, 2>(tq, tk, p, grid, stream);
  return launch_one<kFp8, kMode, kPaged, 1, 1>(tq, tk, p, grid, stream);
}
template <bool kFp8, int kMode>
cudaError_t launch(const CUtensorMap& tq, const CUtensorMap& tk, const ScanParams& p, int grid, cudaStream_t stream) {
  return p.page_table != nullptr ? launch_paged<kFp8, kMode, true>(tq, tk, p, grid, stream)
                                 : launch_paged<kFp8, kMode, false>(tq, tk, p, grid, stream);
}

}  // namespace

namespace {
__global__ void wait_timeout_probe_kernel(unsigned int limit_us, int* result2) {
  __shared__ uint64_t bar;
  __shared__ int abort_flag[2];  // flag, limit in microseconds
  if (threadIdx.x == 0) {
    mbar_init(smem_u32(&bar), 1);
    abort_flag[0] = 0;
    abort_flag[1] = static_cast<int>(limit_us);
    fence_mbar_init();
  }
  __syncthreads();
  // phase 0 of `bar` never completes: the wait can only end by its time limit
  const bool ok = mbar_wait<40>(smem_u32(&bar), 0, abort_flag);
  __syncthreads();
  if (threadIdx.x == 0) {
    result2[0] = ok ? 1 : 0;
    result2[1] = abort_flag[0];
  }
}
}  // namespace

cudaError_t launch_wait_timeout_probe(unsigned int limit_us, int* result2, cudaStream_t stream) {
  wait_timeout_probe_kernel<<<1, 32, 0, stream>>>(limit_us, result2);
  return cudaGetLastError();
}

bool scan_mma_supported(int dtype, int H, int D) {
  return (dtype == LT_DTYPE_BF16 || dtype == LT_DTYPE_E4M3) && H == kH && D == kD;
}

cudaError_t launch_scan_mma(int dtype, int mode, const void* q, int T, const void* k, long long n_keys_view,
                            long long key_pitch_elems, const ScanParams& params, int grid, cudaStream_t stream) {
  ScanParams p = params;
  if (p.wait_limit_us == 0) p.wait_limit_us = kDefaultWaitLimitUs;
  const bool fp8 = (dtype == LT_DTYPE_E4M3);
  const size_t esz = fp8 ? 1 : 2;
  CUtensorMap tq, tk;
  if (!make_map(&tq, fp8, q, static_cast<uint64_t>(T) * kH, kD * esz, 256)) return cudaErrorInvalidValue;
  // dense keys: one 128-row box per tile; paged keys (k = the page pool, n_keys_view = its rows): 64-row boxes
  if (!make_map(&tk, fp8, k, static_cast<uint64_t>(n_keys_view), static_cast<uint64_t>(key_pitch_elems) * esz,
                p.page_table != nullptr ? kPageKeys : 128))
    return cudaErrorInvalidValue;
  if (fp8) {
    return mode == kModeFilter ? launch<true, kModeFilter>(tq, tk, p, grid, stream) : launch<true, kModeDump>(tq, tk, p, grid, stream);
  }
  return mode == kModeFilter ? launch<false, kModeFilter>(tq, tk, p, grid, stream) : launch<false, kModeDump>(tq, tk, p, grid, stream);
}

}  // namespace lt
