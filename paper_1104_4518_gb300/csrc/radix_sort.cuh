// Device radix sort of 64-bit keys and the chained scan that its passes, the
// deduplication and the row tables share.
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

#include "device_common.cuh"
#include "internal.h"

namespace bfsint {

// ---------------- chained scan ----------------
// Tiles of one launch pass their running totals on through one 64-bit word per
// tile (and bin): [63:62] what the word holds, [61:56] the launch's epoch
// (words of another epoch count as empty, so that one cleared array serves
// several launches), [55:0] the value.  A tile takes its number from a ticket,
// so every tile it waits for belongs to a CTA that is already running and
// that publishes before it waits itself.
constexpr uint64_t kTileSum = 1ull << 62;     // the tile's own total
constexpr uint64_t kTilePrefix = 2ull << 62;  // the total of the tile and all before it
constexpr uint64_t kTileValue = (1ull << 56) - 1;
constexpr unsigned kChainSpinLimit = 1u << 22;  // polls of one word (each a round trip to L2): seconds

__device__ __forceinline__ uint64_t tile_word(uint64_t kind, int epoch, uint64_t value) {
  return kind | ((uint64_t)epoch << 56) | value;
}
__device__ __forceinline__ void publish_tile(uint64_t* word, uint64_t kind, int epoch, uint64_t value) {
  asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(word), "l"(tile_word(kind, epoch, value)) : "memory");
}
__device__ __forceinline__ uint64_t load_tile(const uint64_t* word) {
  uint64_t w;
  asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(w) : "l"(word) : "memory");
  return w;
}

// Sum over all tiles before `tile` of the words at state + t * stride, by one
// thread.  Returns false (and posts BFS_ERR_TIMEOUT in *status) when a word
// stays empty for kChainSpinLimit polls or another CTA has posted an error.
// W words are in flight: the tiles resolve themselves at W per round trip to L2
// at best, which has to exceed the rate at which the launch works through them.
template <int W>
__device__ __forceinline__ bool sum_before(const uint64_t* state, long long stride, long long tile, int epoch,
                                           int* status, uint64_t& sum) {
  sum = 0;
  unsigned polls = 0;
  for (long long t = tile - 1; t >= 0;) {
    uint64_t w[W];
#pragma unroll
    for (int j = 0; j < W; ++j) w[j] = t - j >= 0 ? load_tile(state + (t - j) * stride) : tile_word(kTilePrefix, epoch, 0);
    int used = 0;
    bool done = false;
#pragma unroll
    for (int j = 0; j < W; ++j) {
      if (!done && used == j && (w[j] >> 62) != 0 && (int)((w[j] >> 56) & 63u) == epoch) {
        sum += w[j] & kTileValue;
        done = (w[j] & kTilePrefix) != 0;
        used = j + 1;
      }
    }
    if (done) return true;
    t -= used;
    if (used == 0 && ((++polls > kChainSpinLimit) || bfsdev::ld_relaxed_i32(status) != 0)) {
      atomicCAS(status, 0, (int)BFS_ERR_TIMEOUT);
      return false;
    }
  }
  return true;
}

// The same by a whole warp, for one word per tile: 32 words in flight.
__device__ __forceinline__ bool sum_before_warp(const uint64_t* state, long long tile, int epoch, int* status,
                                                uint64_t& sum) {
  const int lane = threadIdx.x & 31;
  sum = 0;
  unsigned polls = 0;
  for (long long t = tile - 1; t >= 0;) {
    const uint64_t w = t - lane >= 0 ? load_tile(state + t - lane) : tile_word(kTilePrefix, epoch, 0);
    const bool full = (w >> 62) != 0 && (int)((w >> 56) & 63u) == epoch;
    const unsigned empty = __ballot_sync(bfsdev::kFull, !full);
    const unsigned prefix = __ballot_sync(bfsdev::kFull, full && (w & kTilePrefix) != 0);
    const int used = empty ? __ffs(empty) - 1 : 32;              // leading words that hold something
    const int stop = prefix ? __ffs(prefix) : 33;                // up to and with the first prefix
    uint64_t v = lane < min(used, stop) ? (w & kTileValue) : 0;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(bfsdev::kFull, v, o);
    sum += v;
    if (stop <= used) return true;
    t -= used;
    if (used == 0) {
      int give_up = 0;
      if (lane == 0) give_up = (++polls > kChainSpinLimit) || bfsdev::ld_relaxed_i32(status) != 0;
      if (__shfl_sync(bfsdev::kFull, give_up, 0)) {
        if (lane == 0) atomicCAS(status, 0, (int)BFS_ERR_TIMEOUT);
        return false;
      }
    }
  }
  return true;
}

// ---------------- sort ----------------
constexpr int kSortThreads = 512;
constexpr int kSortWarps = kSortThreads / 32;
constexpr int kSortItems = 16;
constexpr int kSortTile = kSortThreads * kSortItems;  // 8,192 keys
constexpr int kSortMaxBits = 9;
constexpr int kSortBins = 1 << kSortMaxBits;
constexpr int kSortMaxPasses = 8;

// The digits of a sort on key bits [lo, hi): equal widths of at most kSortMaxBits.
struct SortPlan {
  int passes = 0;
  int shift[kSortMaxPasses] = {};
  int bits[kSortMaxPasses] = {};
};
SortPlan sort_plan(int lo, int hi);

// What a sort of up to cap keys needs beside its two key buffers, all in one
// device block that starts zeroed (sort_scratch_bytes of it).
struct SortScratch {
  unsigned long long* hist = nullptr;  // [passes][kSortBins] digit counts, then their exclusive prefix sums
  unsigned* ticket = nullptr;          // [passes]
  uint64_t* state = nullptr;           // [tiles][kSortBins]
};
size_t sort_scratch_bytes(long long cap);
SortScratch sort_scratch_at(void* block, long long cap);

// Digit histograms of keys[0, N) into sc.hist.
int launch_sort_hist(const uint64_t* keys, long long N, const SortPlan& plan, const SortScratch& sc, cudaStream_t s);
// The passes of a sort of *d_n keys (at most cap; cap itself when d_n is null),
// whose histograms sc.hist holds.  Stable unless it starts at bit 0: keys sorted
// from there on must have no bits above the sorted ones, so that equal keys are
// alike and the first pass need not keep their order.  Nothing is waited for.  Returns the
// buffer that will hold the result; *status receives BFS_ERR_TIMEOUT when a
// wait ran out.
uint64_t* launch_sort_passes(uint64_t* keys, uint64_t* alt, long long cap, const unsigned long long* d_n,
                             const SortPlan& plan, const SortScratch& sc, int* status, cudaStream_t s);

}  // namespace bfsint
