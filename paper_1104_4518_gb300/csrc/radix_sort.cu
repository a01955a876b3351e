// Least-significant-digit radix sort of 64-bit keys, in the manner of the
// published one-sweep method (Adinets and Merrill, 2022): one read for all
// digit histograms, one read and one write per pass, the tiles of a pass linked
// by a chained scan with look-back (Merrill and Garland, 2016).  The order of
// equal digits is kept, except by a pass on bit 0 (see launch_sort_passes).
//
// All digit histograms are taken in one read of the keys (by the caller, who
// often makes the keys anyway), and each pass then reads and writes every key
// once: a tile of 8,192 keys ranks its keys in shared memory, learns where each
// digit's run starts from the tiles before it (chained scan), and writes the
// keys from shared memory in digit order, so that a run of a digit leaves in
// consecutive addresses.  A pass of 134 M keys takes 0.60 ms (the first) to 0.87:
// 0.32 ms of it is the DRAM traffic's due, and what bounds it is the ranking (nine
// ballots and two shared-memory updates per 32 keys).  It took 0.96 ms while the
// fully unrolled scans over the CTA's warps spilled the keys' registers, every key
// of a tile was tested against the end of the input, and the first pass was stable
// too.  The earlier form, with a histogram kernel, a scan and a direct scatter from
// registers per 8-bit digit, took 2.05 ms and a host synchronisation per pass.
// Nine-bit digits sort 44-bit keys in five passes instead of six.
#include <algorithm>

#include "radix_sort.cuh"

namespace bfsint {
namespace {

using bfsdev::kFull;

// Exclusive prefix sum over the CTA's kSortThreads values; s_warp holds kSortWarps.
template <typename T>
__device__ __forceinline__ T cta_exclusive_scan(T x, T* s_warp) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  T incl = x;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const T y = __shfl_up_sync(kFull, incl, o);
    if (lane >= o) incl += y;
  }
  if (lane == 31) s_warp[wid] = incl;
  __syncthreads();
  T before = 0;
#pragma unroll 4
  for (int w = 0; w < kSortWarps; ++w) before += w < wid ? s_warp[w] : 0;
  __syncthreads();
  return before + incl - x;
}

__global__ void __launch_bounds__(kSortThreads) sort_hist_kernel(const uint64_t* __restrict__ keys, long long N,
                                                                 SortPlan plan, unsigned long long* __restrict__ hist) {
  __shared__ unsigned s_h[kSortMaxPasses * kSortBins];
  for (int i = threadIdx.x; i < plan.passes * kSortBins; i += kSortThreads) s_h[i] = 0;
  __syncthreads();
  const long long stride = (long long)gridDim.x * kSortThreads;
  for (long long i = (long long)blockIdx.x * kSortThreads + threadIdx.x; i < N; i += stride) {
    const uint64_t k = keys[i];
#pragma unroll
    for (int q = 0; q < kSortMaxPasses; ++q)
      if (q < plan.passes) atomicAdd(&s_h[q * kSortBins + (int)(k >> plan.shift[q] & ((1u << plan.bits[q]) - 1u))], 1u);
  }
  __syncthreads();
  for (int i = threadIdx.x; i < plan.passes * kSortBins; i += kSortThreads)
    if (s_h[i]) atomicAdd(&hist[i], (unsigned long long)s_h[i]);
}

// Digit counts of a pass (one CTA each) to the start of each digit's run.
__global__ void __launch_bounds__(kSortThreads) sort_base_kernel(unsigned long long* hist) {
  __shared__ unsigned long long s_warp[kSortWarps];
  static_assert(kSortBins == kSortThreads, "one bin per thread");
  unsigned long long* h = hist + blockIdx.x * kSortBins;
  const unsigned long long c = h[threadIdx.x];
  h[threadIdx.x] = cta_exclusive_scan(c, s_warp);
}

constexpr int kChainWords = 4;  // see sum_before; 12 and 24 made a pass 5 % and 27 % slower (L2 traffic)

struct PassArgs {
  const uint64_t* __restrict__ in;
  uint64_t* __restrict__ out;
  const unsigned long long* d_n;
  long long cap;
  int shift, bits, epoch;
  const unsigned long long* base;
  uint64_t* state;
  unsigned* ticket;
  int* status;
};

// kStable: keys of one digit leave in the order they came.  The pass on the lowest
// digit of keys that have no bits below or above the sorted ones need not keep it
// (keys equal in all digits are the same key), and ranks by one shared-memory
// counter per digit: 0.60 ms for 134 M keys, against 0.77.
// In a stable pass the input ends in keys of all ones, which rank behind the real
// keys of the last digit of the last tile: nothing tests for the end before the write.
template <bool kStable>
__global__ void __launch_bounds__(kSortThreads, 2) sort_pass_kernel(PassArgs a) {
  extern __shared__ uint64_t s_keys[];                // kSortTile
  __shared__ __align__(16) unsigned short s_cnt[kStable ? kSortWarps : 2][kSortBins];
  unsigned* const s_count = reinterpret_cast<unsigned*>(&s_cnt[0][0]);  // !kStable: one counter per digit
  __shared__ int s_loc[kSortBins];
  __shared__ long long s_base[kSortBins];
  __shared__ int s_warp[kSortWarps];
  __shared__ unsigned s_tile;
  __shared__ int s_bad;
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  if (tid == 0) {
    s_tile = atomicAdd(a.ticket, 1u);
    s_bad = bfsdev::ld_relaxed_i32(a.status);
  }
  for (int i = tid; i < (int)(sizeof(s_cnt) / sizeof(unsigned)); i += kSortThreads) s_count[i] = 0;
  __syncthreads();
  const long long N = a.d_n ? min((long long)*a.d_n, a.cap) : a.cap;
  const long long tile = s_tile, first = tile * kSortTile;
  if (first >= N || s_bad) return;  // after an error no tile waits for long: see sum_before
  const unsigned dmask = (1u << a.bits) - 1u;

  // keys of the warp, 32 consecutive ones per step; rank of each among its digit's earlier keys of the warp
  uint64_t key[kSortItems];
  unsigned rank[kSortItems / 2];
  const int at = wid * (32 * kSortItems) + lane, left = (int)min((long long)kSortTile, N - first);
  const uint64_t* const in = a.in + first + at;
#pragma unroll
  for (int i = 0; i < kSortItems; ++i) key[i] = at + i * 32 < left ? in[i * 32] : ~0ull;
#pragma unroll
  for (int i = 0; i < kSortItems; ++i) {
    const unsigned d = (unsigned)(key[i] >> a.shift) & dmask;
    unsigned c = 0;
    if constexpr (!kStable) {
      if (at + i * 32 < left) c = atomicAdd(&s_count[d], 1u);
    } else {
      unsigned peers = kFull;
#pragma unroll
      for (int b = 0; b < kSortMaxBits; ++b) {
        const unsigned flip = (d >> b & 1u) - 1u;  // all ones where the bit is clear
        peers &= __ballot_sync(kFull, flip == 0) ^ flip;
      }
      const unsigned before = peers & bfsdev::lanemask_lt();
      c = s_cnt[wid][d];
      __syncwarp();
      if (before == 0) s_cnt[wid][d] = (unsigned short)(c + __popc(peers));
      __syncwarp();
      c += __popc(before);
    }
    if (i & 1) rank[i / 2] |= c << 16;
    else rank[i / 2] = c;
  }
  __syncthreads();
  // thread d: digit d's count in the tile, by warp and in all
  int cnt = 0;
  if constexpr (kStable) {
#pragma unroll 4
    for (int w = 0; w < kSortWarps; ++w) {
      const int c = s_cnt[w][tid];
      s_cnt[w][tid] = (unsigned short)cnt;
      cnt += c;
    }
  } else {
    cnt = (int)s_count[tid];
  }
  uint64_t* mine = a.state + tile * kSortBins + tid;
  publish_tile(mine, tile == 0 ? kTilePrefix : kTileSum, a.epoch, (uint64_t)cnt);
  s_loc[tid] = cta_exclusive_scan(cnt, s_warp);
  __syncthreads();
  // the tile in digit order in shared memory; its keys' registers are free for the words of other tiles
#pragma unroll
  for (int i = 0; i < kSortItems; ++i) {
    if (kStable || at + i * 32 < left) {
      const unsigned d = (unsigned)(key[i] >> a.shift) & dmask;
      s_keys[s_loc[d] + (kStable ? s_cnt[wid][d] : 0) + (int)(rank[i / 2] >> (16 * (i & 1)) & 0xffffu)] = key[i];
    }
  }
  uint64_t before = 0;
  const bool ok = sum_before<kChainWords>(a.state + tid, kSortBins, tile, a.epoch, a.status, before);
  if (ok && tile > 0) publish_tile(mine, kTilePrefix, a.epoch, before + (uint64_t)cnt);
  s_base[tid] = (long long)(a.base[tid] + before) - s_loc[tid];
  if (__syncthreads_or(!ok)) return;  // a wait ran out: write nothing
  for (int i = tid; i < left; i += kSortThreads) {
    const uint64_t k = s_keys[i];
    a.out[s_base[(unsigned)(k >> a.shift) & dmask] + i] = k;
  }
}

constexpr size_t kSortDynSmem = sizeof(uint64_t) * kSortTile;

long long sort_tiles(long long cap) { return (cap + kSortTile - 1) / kSortTile; }

}  // namespace

SortPlan sort_plan(int lo, int hi) {
  SortPlan p;
  const int total = hi - lo;
  p.passes = (total + kSortMaxBits - 1) / kSortMaxBits;
  for (int q = 0, at = lo; q < p.passes; ++q) {
    p.shift[q] = at;
    p.bits[q] = (hi - at + (p.passes - q) - 1) / (p.passes - q);
    at += p.bits[q];
  }
  return p;
}

size_t sort_scratch_bytes(long long cap) {
  return sizeof(unsigned long long) * kSortMaxPasses * kSortBins + 256 +
         sizeof(uint64_t) * kSortBins * (size_t)std::max(1ll, sort_tiles(cap));
}

SortScratch sort_scratch_at(void* block, long long cap) {
  (void)cap;
  SortScratch sc;
  char* p = static_cast<char*>(block);
  sc.hist = reinterpret_cast<unsigned long long*>(p);
  p += sizeof(unsigned long long) * kSortMaxPasses * kSortBins;
  sc.ticket = reinterpret_cast<unsigned*>(p);
  sc.state = reinterpret_cast<uint64_t*>(p + 256);
  return sc;
}

int launch_sort_hist(const uint64_t* keys, long long N, const SortPlan& plan, const SortScratch& sc, cudaStream_t s) {
  DeviceInfo di;
  if (int e = current_device_info(&di)) return e;
  const long long grid = std::min<long long>(2 * di.sm_count, (N + kSortTile - 1) / kSortTile);
  if (grid > 0) sort_hist_kernel<<<(unsigned)grid, kSortThreads, 0, s>>>(keys, N, plan, sc.hist);
  BFS_CUDA_TRY(cudaGetLastError());
  return BFS_OK;
}

uint64_t* launch_sort_passes(uint64_t* keys, uint64_t* alt, long long cap, const unsigned long long* d_n,
                             const SortPlan& plan, const SortScratch& sc, int* status, cudaStream_t s) {
  if (cap <= 0 || plan.passes == 0) return keys;
  for (const void* f : {(const void*)sort_pass_kernel<false>, (const void*)sort_pass_kernel<true>})
    cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSortDynSmem);
  sort_base_kernel<<<plan.passes, kSortThreads, 0, s>>>(sc.hist);
  for (int q = 0; q < plan.passes; ++q) {
    PassArgs a{keys, alt, d_n, cap, plan.shift[q], plan.bits[q], q + 1, sc.hist + q * kSortBins, sc.state, sc.ticket + q,
               status};
    // from bit 0 on, the callers' keys have no bits beside the sorted ones
    const auto pass = plan.shift[q] == 0 ? sort_pass_kernel<false> : sort_pass_kernel<true>;
    pass<<<(unsigned)sort_tiles(cap), kSortThreads, kSortDynSmem, s>>>(a);
    std::swap(keys, alt);
  }
  return keys;
}

int radix_sort_u64(uint64_t* keys, uint64_t* alt, long long N, int lo_bit, int hi_bit, cudaStream_t s,
                   uint64_t** sorted) {
  *sorted = keys;
  if (N <= 0 || lo_bit >= hi_bit) return BFS_OK;
  const SortPlan plan = sort_plan(lo_bit, hi_bit);
  const size_t bytes = sort_scratch_bytes(N) + 256;
  char* block = nullptr;
  if (int e = dev_alloc((void**)&block, bytes, "radix sort tiles")) return e;
  int* status = reinterpret_cast<int*>(block + bytes - 256);
  const SortScratch sc = sort_scratch_at(block, N);
  int st[4] = {0, 0, 0, 0};
  cudaError_t err = cudaMemsetAsync(block, 0, bytes, s);
  int rc = err == cudaSuccess ? launch_sort_hist(keys, N, plan, sc, s) : BFS_OK;
  if (err == cudaSuccess && !rc) {
    *sorted = launch_sort_passes(keys, alt, N, nullptr, plan, sc, status, s);
    err = cudaGetLastError();
  }
  if (err == cudaSuccess && !rc) err = cudaMemcpyAsync(st, status, sizeof(st), cudaMemcpyDeviceToHost, s);
  if (err == cudaSuccess) err = cudaStreamSynchronize(s);
  dev_free(block);
  if (rc) return rc;
  if (err != cudaSuccess) return cuda_fail(err, "radix sort");
  if (st[0]) return fail(st[0], "radix sort: " + device_status_message(st));
  return BFS_OK;
}

}  // namespace bfsint
