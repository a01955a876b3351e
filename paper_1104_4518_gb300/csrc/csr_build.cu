// Edge list -> symmetric, deduplicated, row-sorted CSR on the device, the row
// tables that a graph keeps beside it, and the CSR validation used by
// bfs_graph_create(BFS_VALIDATE).
//
// The paper stores each undirected edge in both rows with every row sorted
// (Sec. 4.1) and its benchmark symmetrises the generated edges (Sec. 6).  Here:
//   1. every non-loop edge (u, v) emits the keys (u << b) | v and (v << b) | u,
//      b = bits of n - 1, appended a tile at a time, and the digit histograms of
//      all sort passes are counted on the way;
//   2. the keys are sorted on their 2b significant bits (radix_sort.cu);
//   3. a key equal to its predecessor is a repeat; one pass with a chained scan
//      of the "first of its value" flags gives every kept key its slot and
//      writes its column (the low b bits), and the row changes between
//      consecutive keys give the int64 row offsets.
// Nothing is read back before step 3 is enqueued: the number of keys stays on
// the device.  The host waits twice, for the entry count and at the end.
#include <algorithm>
#include <cstdio>

#include "device_common.cuh"
#include "internal.h"
#include "radix_sort.cuh"

namespace bfsint {
namespace {

using bfsdev::kFull;

constexpr int kScanThreads = 512;
constexpr int kScanItems = 8;
constexpr int kScanTile = kScanThreads * kScanItems;

// What the construction kernels report; one block, cleared before them and read back after.
struct BuildReport {
  unsigned long long nkeys;  // keys emitted
  unsigned long long nnz;    // keys kept
  unsigned long long nlive;  // rows with entries
  unsigned long long nbig;   // chunks of rows longer than kChunkEdges
  int status[4];             // device status (BFS_ERR_TIMEOUT of a chained scan)
  int bad;                   // an edge endpoint outside [0, n)
  unsigned ticket;           // tiles handed out by the chained scan of this block's kernel
};

// ---------------- key emission ----------------
constexpr int kKeyThreads = 256;
constexpr int kKeyWarps = kKeyThreads / 32;
constexpr int kKeyItems = 8;
constexpr int kKeyTile = kKeyThreads * kKeyItems;  // 2,048 edges

// Keys of the arcs of edge e = (u, v): mode 0 (undirected) emits u -> v and
// v -> u, mode 1 u -> v only, mode 2 v -> u only (the transpose).  A tile's
// keys take their places with one atomic (one per warp and step on the same
// word made this kernel 1.48 ms for 67 M edges), in any order: the sort orders
// them, and equal keys are alike.  0.36 ms for 67 M edges, 0.24 of them the DRAM
// traffic's due; 0.62 while the plan was indexed at run time, from a local copy.
__global__ void __launch_bounds__(kKeyThreads) make_keys_kernel(const int32_t* __restrict__ src,
                                                                const int32_t* __restrict__ dst, int64_t m, int32_t n,
                                                                int vbits, int mode, SortPlan plan,
                                                                uint64_t* __restrict__ keys,
                                                                unsigned long long* __restrict__ hist,
                                                                BuildReport* __restrict__ rep) {
  __shared__ unsigned s_h[kSortMaxPasses * kSortBins];
  __shared__ int s_cnt[kKeyItems * kKeyWarps];  // valid edges of each step and warp, then their exclusive sums
  __shared__ unsigned long long s_at;
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const int per = mode == 0 ? 2 : 1;
  for (int i = tid; i < plan.passes * kSortBins; i += kKeyThreads) s_h[i] = 0;
  __syncthreads();
  auto count = [&](uint64_t k) {
#pragma unroll
    for (int q = 0; q < kSortMaxPasses; ++q)
      if (q < plan.passes) atomicAdd(&s_h[q * kSortBins + (int)(k >> plan.shift[q] & ((1u << plan.bits[q]) - 1u))], 1u);
  };
  for (long long base = (long long)blockIdx.x * kKeyTile; base < m; base += (long long)gridDim.x * kKeyTile) {
    int u[kKeyItems], v[kKeyItems];
    unsigned bm[kKeyItems];
    bool out = false;
#pragma unroll
    for (int i = 0; i < kKeyItems; ++i) {
      const long long e = base + i * kKeyThreads + tid;
      u[i] = e < m ? __ldg(&src[e]) : 0;
      v[i] = e < m ? __ldg(&dst[e]) : 0;
    }
#pragma unroll
    for (int i = 0; i < kKeyItems; ++i) {
      const bool in = (unsigned)u[i] < (unsigned)n && (unsigned)v[i] < (unsigned)n;
      out |= !in;
      bm[i] = __ballot_sync(kFull, in && u[i] != v[i]);  // an edge past m reads as the loop (0, 0)
      if (lane == 0) s_cnt[i * kKeyWarps + wid] = __popc(bm[i]);
    }
    if (out) atomicExch(&rep->bad, 1);
    __syncthreads();
    if (wid == 0) {  // exclusive sums over the 64 counts, two per lane
      const int c0 = s_cnt[2 * lane], c1 = s_cnt[2 * lane + 1];
      int incl = c0 + c1;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(kFull, incl, o);
        if (lane >= o) incl += y;
      }
      s_cnt[2 * lane] = incl - c0 - c1;
      s_cnt[2 * lane + 1] = incl - c1;
      if (lane == 31) s_at = incl ? atomicAdd(&rep->nkeys, (unsigned long long)(per * incl)) : 0ull;
    }
    __syncthreads();
    const unsigned long long at = s_at;
#pragma unroll
    for (int i = 0; i < kKeyItems; ++i) {
      if (!((bm[i] >> lane) & 1u)) continue;
      const long long pos = (long long)at + (long long)per * (s_cnt[i * kKeyWarps + wid] + __popc(bm[i] & bfsdev::lanemask_lt()));
      const uint64_t fwd = ((uint64_t)u[i] << vbits) | (uint64_t)v[i], rev = ((uint64_t)v[i] << vbits) | (uint64_t)u[i];
      if (mode == 0) {
        reinterpret_cast<ulonglong2*>(keys)[pos >> 1] = make_ulonglong2(fwd, rev);  // pos is even
        count(fwd);
        count(rev);
      } else {
        keys[pos] = mode == 1 ? fwd : rev;
        count(mode == 1 ? fwd : rev);
      }
    }
    __syncthreads();
  }
  __syncthreads();
  for (int i = tid; i < plan.passes * kSortBins; i += kKeyThreads)
    if (s_h[i]) atomicAdd(&hist[i], (unsigned long long)s_h[i]);
}
static_assert(kKeyItems * kKeyWarps == 64, "the scan of the counts covers two per lane");

// ---------------- exclusive scan (int64 output) ----------------
// Input element i is in[i] (uint32 or int64 source).
struct ScanInput {
  const uint32_t* u32 = nullptr;
  const int64_t* i64 = nullptr;
  __device__ __forceinline__ long long at(long long i) const { return u32 ? (long long)u32[i] : (long long)i64[i]; }
};

__device__ __forceinline__ long long block_scan_ll(long long x, long long* s_warp, long long& total) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  long long incl = x;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const long long y = __shfl_up_sync(kFull, incl, o);
    if (lane >= o) incl += y;
  }
  if (lane == 31) s_warp[wid] = incl;
  __syncthreads();
  if (wid == 0) {
    const int nw = blockDim.x / 32;
    long long v = lane < nw ? s_warp[lane] : 0;
    long long inc = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const long long y = __shfl_up_sync(kFull, inc, o);
      if (lane >= o) inc += y;
    }
    if (lane < nw) s_warp[lane] = inc - v;
    if (lane == nw - 1) s_warp[32] = inc;
  }
  __syncthreads();
  const long long excl = s_warp[wid] + incl - x;
  total = s_warp[32];
  __syncthreads();
  return excl;
}

// Tile sums.
__global__ void scan_reduce_kernel(ScanInput in, long long N, int64_t* __restrict__ sums) {
  __shared__ long long s_warp[33];
  const long long base = (long long)blockIdx.x * kScanTile;
  long long x = 0;
#pragma unroll
  for (int i = 0; i < kScanItems; ++i) {
    const long long idx = base + (long long)threadIdx.x * kScanItems + i;
    if (idx < N) x += in.at(idx);
  }
  long long total;
  block_scan_ll(x, s_warp, total);
  if (threadIdx.x == 0) sums[blockIdx.x] = total;
}

// Exclusive scan of each tile plus its tile offset.
__global__ void scan_down_kernel(ScanInput in, long long N, const int64_t* __restrict__ tile_off,
                                 int64_t* __restrict__ out) {
  __shared__ long long s_warp[33];
  const long long base = (long long)blockIdx.x * kScanTile;
  long long vals[kScanItems];
  long long x = 0;
#pragma unroll
  for (int i = 0; i < kScanItems; ++i) {
    const long long idx = base + (long long)threadIdx.x * kScanItems + i;
    vals[i] = idx < N ? in.at(idx) : 0;
    x += vals[i];
  }
  long long total;
  long long run = block_scan_ll(x, s_warp, total) + (tile_off ? tile_off[blockIdx.x] : 0);
#pragma unroll
  for (int i = 0; i < kScanItems; ++i) {
    const long long idx = base + (long long)threadIdx.x * kScanItems + i;
    if (idx < N) out[idx] = run;
    run += vals[i];
  }
}

// Exclusive scan of N elements into out (int64); returns the total in *total (host).
int exclusive_scan(const ScanInput& in, long long N, int64_t* out, cudaStream_t s, long long* total) {
  if (N <= 0) {
    *total = 0;
    return BFS_OK;
  }
  const long long tiles = (N + kScanTile - 1) / kScanTile;
  int64_t* sums = nullptr;
  int64_t* sums_off = nullptr;
  if (tiles > 1) {
    if (int e = dev_alloc((void**)&sums, sizeof(int64_t) * tiles, "scan tile sums")) return e;
    if (int e = dev_alloc((void**)&sums_off, sizeof(int64_t) * tiles, "scan tile offsets")) {
      dev_free(sums);
      return e;
    }
    scan_reduce_kernel<<<(unsigned)tiles, kScanThreads, 0, s>>>(in, N, sums);
    ScanInput si;
    si.i64 = sums;
    long long t2 = 0;
    if (int e = exclusive_scan(si, tiles, sums_off, s, &t2)) {
      dev_free(sums);
      dev_free(sums_off);
      return e;
    }
  }
  scan_down_kernel<<<(unsigned)tiles, kScanThreads, 0, s>>>(in, N, sums_off, out);
  cudaError_t err = cudaGetLastError();
  // total = out[N-1] + in[N-1]
  long long last_out = 0, last_in = 0;
  if (err == cudaSuccess) err = cudaMemcpyAsync(&last_out, out + (N - 1), sizeof(long long), cudaMemcpyDeviceToHost, s);
  if (err == cudaSuccess) {
    if (in.u32) {
      uint32_t v = 0;
      err = cudaMemcpyAsync(&v, in.u32 + (N - 1), sizeof(v), cudaMemcpyDeviceToHost, s);
      if (err == cudaSuccess) err = cudaStreamSynchronize(s);
      last_in = v;
    } else {
      err = cudaMemcpyAsync(&last_in, in.i64 + (N - 1), sizeof(long long), cudaMemcpyDeviceToHost, s);
      if (err == cudaSuccess) err = cudaStreamSynchronize(s);
    }
  }
  if (sums) dev_free(sums);
  if (sums_off) dev_free(sums_off);
  if (err != cudaSuccess) return cuda_fail(err, "exclusive scan");
  *total = last_out + last_in;
  return BFS_OK;
}

// ---------------- dedup + CSR emission ----------------
constexpr int kEmitThreads = 512;
constexpr int kEmitWarps = kEmitThreads / 32;
constexpr int kEmitItems = 16;
constexpr int kEmitTile = kEmitThreads * kEmitItems;  // 8,192 keys

// One read of the sorted keys: every key that differs from its predecessor is
// kept, its slot is the number of kept keys before it (within the warp's 512
// consecutive keys by ballots, across tiles by a chained scan), and where its
// row differs from the predecessor's the rows in between start at that slot.
// 134 M keys: 0.60 ms, 0.24 of them the
// DRAM traffic's due (a flag scan and an emission kernel took 1.7 ms; with 64-bit
// end tests and four shuffles per key and step 0.72).
__global__ void __launch_bounds__(kEmitThreads, 2) emit_csr_kernel(const uint64_t* __restrict__ keys, int vbits, int32_t n,
                                                                int64_t* __restrict__ off, int32_t* __restrict__ adj,
                                                                uint64_t* __restrict__ state, BuildReport* rep) {
  __shared__ int s_cnt[kEmitWarps];
  __shared__ unsigned s_tile;
  __shared__ unsigned long long s_at;
  __shared__ int s_ok;
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  if (tid == 0) {
    s_tile = atomicAdd(&rep->ticket, 1u);
    s_ok = bfsdev::ld_relaxed_i32(rep->status) == 0;
  }
  __syncthreads();
  const long long N = (long long)rep->nkeys, tile = s_tile, seg = tile * kEmitTile + wid * (32 * kEmitItems);
  if (tile * kEmitTile >= N || !s_ok) return;
  const uint64_t vmask = (1ull << vbits) - 1ull;
  const int left = (int)max(0ll, min(32ll * kEmitItems, N - seg));  // the warp's keys
  uint64_t key[kEmitItems];
#pragma unroll
  for (int i = 0; i < kEmitItems; ++i) key[i] = i * 32 + lane < left ? keys[seg + i * 32 + lane] : 0;
  uint64_t before = ~0ull;  // the key before the warp's first
  if (seg > 0 && seg < N) before = keys[seg - 1];
  unsigned kept[kEmitItems];
  int cnt = 0;
  uint64_t carry = before;  // lane 0's predecessor
#pragma unroll
  for (int i = 0; i < kEmitItems; ++i) {
    const uint64_t turned = __shfl_sync(kFull, key[i], (lane + 31) & 31);
    const uint64_t prev = lane == 0 ? carry : turned;
    carry = turned;
    kept[i] = __ballot_sync(kFull, i * 32 + lane < left && key[i] != prev);
    cnt += __popc(kept[i]);
  }
  if (lane == 0) s_cnt[wid] = cnt;
  __syncthreads();
  int warp_at = 0, total = 0;
#pragma unroll
  for (int w = 0; w < kEmitWarps; ++w) {
    warp_at += w < wid ? s_cnt[w] : 0;
    total += s_cnt[w];
  }
  if (wid == 0) {
    if (lane == 0) publish_tile(state + tile, tile == 0 ? kTilePrefix : kTileSum, 1, (uint64_t)total);
    uint64_t sum = 0;
    const bool ok = sum_before_warp(state, tile, 1, rep->status, sum);
    if (lane == 0) {
      if (ok && tile > 0) publish_tile(state + tile, kTilePrefix, 1, sum + (uint64_t)total);
      s_ok = ok;
      s_at = sum;
    }
  }
  __syncthreads();
  if (!s_ok) return;
  long long at = (long long)s_at + warp_at;
  int carry_row = seg > 0 ? (int)(before >> vbits) : -1;
#pragma unroll
  for (int i = 0; i < kEmitItems; ++i) {
    const int row = (int)(key[i] >> vbits), turned = __shfl_sync(kFull, row, (lane + 31) & 31);
    const int prev = lane == 0 ? carry_row : turned;
    carry_row = turned;
    const long long pos = at + __popc(kept[i] & bfsdev::lanemask_lt());
    const bool first = (kept[i] >> lane) & 1u;
    if (first) {
      adj[pos] = (int32_t)(key[i] & vmask);
      for (int r = prev + 1; r <= row; ++r) off[r] = pos;
    }
    if (seg + i * 32 + lane == N - 1) {  // the rows after the last key's end with it
      rep->nnz = (unsigned long long)(pos + (first ? 1 : 0));
      for (long long r = row + 1; r <= n; ++r) off[r] = pos + (first ? 1 : 0);
    }
    at += __popc(kept[i]);
  }
}

// ---------------- validation ----------------
__global__ void validate_kernel(const int64_t* __restrict__ off, const int32_t* __restrict__ adj, int32_t n,
                                long long nnz, int symmetric, int* __restrict__ bad) {
  const int lane = threadIdx.x & 31;
  const long long gw = ((long long)blockIdx.x * blockDim.x + threadIdx.x) / 32;
  const long long nwarps = (long long)gridDim.x * blockDim.x / 32;
  if (gw == 0 && lane == 0 && (off[0] != 0 || off[n] != nnz)) atomicExch(bad, 1);
  for (long long u = gw; u < n; u += nwarps) {
    const long long b = off[u], e = off[u + 1];
    if (b > e || b < 0 || e > nnz) {
      if (lane == 0) atomicExch(bad, 2);
      continue;
    }
    for (long long j = b + lane; j < e; j += 32) {
      const int v = adj[j];
      if (v < 0 || v >= n || v == u || (j + 1 < e && adj[j + 1] <= v)) {
        atomicExch(bad, 3);
        continue;
      }
      if (!symmetric) continue;
      // symmetry: u must appear in v's row (binary search; v's row is checked by its own warp)
      long long lo = off[v], hi = off[v + 1];
      if (lo < 0 || hi > nnz || lo > hi) {
        atomicExch(bad, 4);
        continue;
      }
      bool found = false;
      while (lo < hi) {
        const long long mid = (lo + hi) >> 1;
        const int x = adj[mid];
        if (x == u) {
          found = true;
          break;
        }
        if (x < u) lo = mid + 1;
        else hi = mid;
      }
      if (!found) atomicExch(bad, 5);
    }
  }
}

// Row offsets non-decreasing from 0 to nnz (every row inside [0, nnz)).
__global__ void offsets_kernel(const int64_t* __restrict__ off, int32_t n, long long nnz, int* __restrict__ bad) {
  const long long stride = (long long)gridDim.x * blockDim.x;
  const long long i0 = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i0 == 0 && (off[0] != 0 || off[n] != nnz)) atomicExch(bad, 1);
  for (long long v = i0; v < n; v += stride)
    if (off[v] > off[v + 1]) atomicExch(bad, 1);
}

__global__ void shift_kernel(int64_t* off, int32_t* adj, long long n_part, long long nnz_part, long long off_shift,
                             int32_t id_shift) {
  const long long stride = (long long)gridDim.x * blockDim.x;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n_part; i += stride) off[i] += off_shift;
  for (long long j = (long long)blockIdx.x * blockDim.x + threadIdx.x; j < nnz_part; j += stride) adj[j] += id_shift;
}

// ---------------- row tables ----------------
constexpr int kMetaThreads = 512;
constexpr int kMetaWarps = kMetaThreads / 32;
constexpr int kMetaTile = kMetaThreads;  // bitmap words per CTA: 32 per warp, lane j keeps word j

// Per bitmap word: its vertices without entries (`dead`, tail bits set) and the
// number of rows with entries before it (`rank`); in all, the rows with entries
// and the chunks of long rows.
__global__ void __launch_bounds__(kMetaThreads) row_meta_kernel(const int64_t* __restrict__ off, int32_t n,
                                                                long long nwords, uint32_t* __restrict__ dead,
                                                                uint32_t* __restrict__ rank, uint64_t* __restrict__ state,
                                                                BuildReport* rep) {
  __shared__ int s_cnt[kMetaWarps];
  __shared__ unsigned s_tile;
  __shared__ unsigned long long s_at;
  __shared__ int s_ok;
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  if (tid == 0) s_tile = atomicAdd(&rep->ticket, 1u);
  __syncthreads();
  const long long tile = s_tile, w0 = tile * kMetaTile + wid * 32;
  uint32_t live = 0;
  unsigned long long big = 0;
#pragma unroll 8
  for (int j = 0; j < 32; ++j) {
    const long long v = (w0 + j) * 32 + lane;
    const long long d = v < n ? off[v + 1] - off[v] : 0;
    const uint32_t m = __ballot_sync(kFull, d > 0);
    if (lane == j) live = m;
    if (d > kChunkEdges) big += (unsigned long long)((d + kChunkEdges - 1) / kChunkEdges);
  }
  if (big) atomicAdd(&rep->nbig, big);
  const int c = __popc(live);
  int incl = c;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(kFull, incl, o);
    if (lane >= o) incl += y;
  }
  if (lane == 31) s_cnt[wid] = incl;
  __syncthreads();
  int warp_at = 0, total = 0;
#pragma unroll
  for (int w = 0; w < kMetaWarps; ++w) {
    warp_at += w < wid ? s_cnt[w] : 0;
    total += s_cnt[w];
  }
  if (wid == 0) {
    if (lane == 0) publish_tile(state + tile, tile == 0 ? kTilePrefix : kTileSum, 1, (uint64_t)total);
    uint64_t sum = 0;
    const bool ok = sum_before_warp(state, tile, 1, rep->status, sum);
    if (lane == 0) {
      if (ok && tile > 0) publish_tile(state + tile, kTilePrefix, 1, sum + (uint64_t)total);
      if ((tile + 1) * kMetaTile >= nwords) rep->nlive = sum + (uint64_t)total;
      s_ok = ok;
      s_at = sum;
    }
  }
  __syncthreads();
  const long long w = w0 + lane;
  if (!s_ok || w >= nwords) return;
  dead[w] = ~live;
  rank[w] = (uint32_t)(s_at + warp_at + incl - c);
}

// Probe records of the rows with entries (out non-null): one warp per bitmap
// word, packed in id order; and the chunk items of rows longer than kChunkEdges,
// in any order.  A row outside [0, nnz) (a malformed CSR, taken without
// validation) gives a record without entries: creating a graph reads no entry
// that is not there.
__global__ void row_records_kernel(const int64_t* __restrict__ off, const int32_t* __restrict__ adj, long long nnz,
                                   const uint32_t* __restrict__ dead, const uint32_t* __restrict__ rank,
                                   long long nwords, int4* __restrict__ out, int64_t* __restrict__ big,
                                   unsigned long long* big_count) {
  const int lane = threadIdx.x & 31;
  const long long stride = (long long)gridDim.x * blockDim.x / 32;
  for (long long w = ((long long)blockIdx.x * blockDim.x + threadIdx.x) / 32; w < nwords; w += stride) {
    const uint32_t live = ~dead[w];  // the bits past n are dead
    if (!((live >> lane) & 1u)) continue;
    const long long v = w * 32 + lane, b = off[v], e = off[v + 1], d = e - b;
    if (out) {
      const bool in = b >= 0 && e <= nnz;
      out[(long long)rank[w] + __popc(live & bfsdev::lanemask_lt())] =
          make_int4((int)d, in ? adj[e - 1] : 0, in && d > 1 ? adj[e - 2] : 0, in && d > 2 ? adj[e - 3] : 0);
    }
    if (d > kChunkEdges) {
      const unsigned long long nch = (unsigned long long)((d + kChunkEdges - 1) / kChunkEdges);
      const unsigned long long pos = atomicAdd(big_count, nch);
      for (unsigned long long c = 0; c < nch; ++c) big[pos + c] = (v << 32) | (long long)c;
    }
  }
}

// src[j] = u for every entry j of row u (one warp per row; entries outside
// [0, nnz) of a malformed CSR are skipped).
__global__ void expand_rows_kernel(const int64_t* __restrict__ off, int32_t n, long long nnz,
                                   int32_t* __restrict__ src) {
  const int lane = threadIdx.x & 31;
  const long long gw = ((long long)blockIdx.x * blockDim.x + threadIdx.x) / 32;
  const long long nwarps = (long long)gridDim.x * blockDim.x / 32;
  for (long long u = gw; u < n; u += nwarps) {
    const long long b = max((long long)off[u], 0ll), e = min((long long)off[u + 1], nnz);
    for (long long j = b + lane; j < e; j += 32) src[j] = (int32_t)u;
  }
}

int bits_for(int32_t n) {
  int b = 1;
  while (b < 31 && ((int64_t)1 << b) < (int64_t)n) ++b;
  return b;
}

}  // namespace

int exclusive_scan_u32(const uint32_t* in, long long N, int64_t* out, cudaStream_t s, long long* total) {
  ScanInput si;
  si.u32 = in;
  return exclusive_scan(si, N, out, s, total);
}

int build_csr_from_edges(const int32_t* d_src, const int32_t* d_dst, int64_t m, int32_t n, int mode,
                         cudaStream_t s, int64_t** d_off_out, int32_t** d_adj_out, int64_t* nnz_out) {
  DeviceInfo di;
  if (int e = current_device_info(&di)) return e;
  const int vbits = bits_for(n);
  const SortPlan plan = sort_plan(0, 2 * vbits);
  const long long cap = (mode == 0 ? 2 : 1) * (long long)m;
  const long long emit_tiles = (cap + kEmitTile - 1) / kEmitTile;
  // one scratch block: report | sort tables | emission tiles (all cleared) | keys | alternate keys
  const size_t rep_bytes = 256, sort_bytes = (sort_scratch_bytes(cap) + 255) / 256 * 256;
  const size_t emit_bytes = (sizeof(uint64_t) * (size_t)emit_tiles + 255) / 256 * 256;
  const size_t key_bytes = (sizeof(uint64_t) * (size_t)cap + 255) / 256 * 256;
  char* block = nullptr;
  int64_t* off = nullptr;
  int32_t* adj = nullptr;
  BuildReport rep{};
  auto give_up = [&](int rc) {
    if (block) dev_free(block);
    if (off) dev_free(off);
    if (adj) dev_free(adj);
    return rc;
  };
  if (int e = dev_alloc((void**)&off, sizeof(int64_t) * ((size_t)n + 1), "CSR offsets")) return give_up(e);
  uint64_t* sorted = nullptr;
  if (cap > 0) {
    if (int e = dev_alloc((void**)&block, rep_bytes + sort_bytes + emit_bytes + 2 * key_bytes, "sort keys")) return give_up(e);
    BuildReport* d_rep = reinterpret_cast<BuildReport*>(block);
    const SortScratch sc = sort_scratch_at(block + rep_bytes, cap);
    uint64_t* tiles = reinterpret_cast<uint64_t*>(block + rep_bytes + sort_bytes);
    uint64_t* keys = reinterpret_cast<uint64_t*>(block + rep_bytes + sort_bytes + emit_bytes);
    uint64_t* alt = reinterpret_cast<uint64_t*>(reinterpret_cast<char*>(keys) + key_bytes);
    cudaError_t err = cudaMemsetAsync(block, 0, rep_bytes + sort_bytes + emit_bytes, s);
    if (err == cudaSuccess) {
      const long long key_tiles = (m + kKeyTile - 1) / kKeyTile;
      make_keys_kernel<<<(unsigned)std::min<long long>(key_tiles, 4ll * di.sm_count), kKeyThreads, 0, s>>>(
          d_src, d_dst, m, n, vbits, mode, plan, keys, sc.hist, d_rep);
      sorted = launch_sort_passes(keys, alt, cap, &d_rep->nkeys, plan, sc, d_rep->status, s);
      // the columns go to the free key buffer until their number is known
      emit_csr_kernel<<<(unsigned)emit_tiles, kEmitThreads, 0, s>>>(
          sorted, vbits, n, off, reinterpret_cast<int32_t*>(sorted == keys ? alt : keys), tiles, d_rep);
      err = cudaGetLastError();
    }
    if (err == cudaSuccess) err = cudaMemcpyAsync(&rep, d_rep, sizeof(rep), cudaMemcpyDeviceToHost, s);
    if (err == cudaSuccess) err = cudaStreamSynchronize(s);
    if (err != cudaSuccess) return give_up(cuda_fail(err, "CSR construction"));
    if (rep.status[0]) return give_up(fail(rep.status[0], "CSR construction: " + device_status_message(rep.status)));
    if (rep.bad) return give_up(fail(BFS_ERR_INVALID_ARG, "edge endpoint outside [0, n)"));
    if (int e = dev_alloc((void**)&adj, sizeof(int32_t) * (size_t)std::max(1ull, rep.nnz), "CSR adjacency")) return give_up(e);
    if (rep.nnz > 0)
      err = cudaMemcpyAsync(adj, sorted == keys ? alt : keys, sizeof(int32_t) * (size_t)rep.nnz, cudaMemcpyDeviceToDevice, s);
    if (err != cudaSuccess) return give_up(cuda_fail(err, "CSR construction"));
  } else if (int e = dev_alloc((void**)&adj, sizeof(int32_t), "CSR adjacency")) {
    return give_up(e);
  }
  if (rep.nkeys == 0) {  // no key: the emission wrote no offset
    cudaError_t err = cudaMemsetAsync(off, 0, sizeof(int64_t) * ((size_t)n + 1), s);
    if (err != cudaSuccess) return give_up(cuda_fail(err, "CSR construction"));
  }
  cudaError_t err = cudaStreamSynchronize(s);
  if (err != cudaSuccess) return give_up(cuda_fail(err, "CSR construction"));
  if (block) dev_free(block);
  *d_off_out = off;
  *d_adj_out = adj;
  *nnz_out = (int64_t)rep.nnz;
  return BFS_OK;
}

int build_row_tables(const int64_t* d_off, const int32_t* d_adj, int32_t n, int64_t nnz, cudaStream_t s, RowTables* out) {
  DeviceInfo di;
  if (int e = current_device_info(&di)) return e;
  *out = RowTables{};
  const long long nwords = ((long long)n + 31) / 32, tiles = (nwords + kMetaTile - 1) / kMetaTile;
  const size_t word_bytes = (sizeof(uint32_t) * (size_t)nwords + 255) / 256 * 256;
  RowTables t;
  char* scratch = nullptr;
  if (int e = dev_alloc((void**)&t.dead, 2 * word_bytes, "row bitmaps")) return e;
  t.rank = reinterpret_cast<uint32_t*>(reinterpret_cast<char*>(t.dead) + word_bytes);
  BuildReport rep{};
  auto give_up = [&](int rc) {
    if (scratch) dev_free(scratch);
    if (t.probe) dev_free(t.probe);
    if (t.big) dev_free(t.big);
    dev_free(t.dead);
    return rc;
  };
  const size_t bytes = 256 + sizeof(uint64_t) * (size_t)tiles;
  if (int e = dev_alloc((void**)&scratch, bytes, "row table tiles")) return give_up(e);
  BuildReport* d_rep = reinterpret_cast<BuildReport*>(scratch);
  cudaError_t err = cudaMemsetAsync(scratch, 0, bytes, s);
  if (err == cudaSuccess) {
    row_meta_kernel<<<(unsigned)tiles, kMetaThreads, 0, s>>>(d_off, n, nwords, t.dead, t.rank,
                                                             reinterpret_cast<uint64_t*>(scratch + 256), d_rep);
    err = cudaGetLastError();
  }
  if (err == cudaSuccess) err = cudaMemcpyAsync(&rep, d_rep, sizeof(rep), cudaMemcpyDeviceToHost, s);
  if (err == cudaSuccess) err = cudaStreamSynchronize(s);
  if (err != cudaSuccess) return give_up(cuda_fail(err, "row tables"));
  if (rep.status[0]) return give_up(fail(rep.status[0], "row tables: " + device_status_message(rep.status)));
  t.nbig = (int64_t)rep.nbig;
  if (t.nbig > 0)
    if (int e = dev_alloc((void**)&t.big, sizeof(int64_t) * (size_t)t.nbig, "high-degree row chunks")) return give_up(e);
  // the pull works without probe records, only slower: a graph that leaves no room for them does without
  if (dev_alloc((void**)&t.probe, sizeof(int4) * (size_t)std::max(1ull, rep.nlive), "probe records") != BFS_OK)
    t.probe = nullptr;
  row_records_kernel<<<di.sm_count * 8, 256, 0, s>>>(d_off, d_adj, nnz, t.dead, t.rank, nwords, t.probe, t.big, &d_rep->nkeys);
  err = cudaGetLastError();
  if (err == cudaSuccess) err = cudaStreamSynchronize(s);
  if (err != cudaSuccess) return give_up(cuda_fail(err, "row tables"));
  dev_free(scratch);
  *out = t;
  return BFS_OK;
}

int union_shift(int64_t* off, int32_t* adj, int64_t n_part, int64_t nnz_part, int64_t off_shift, int32_t id_shift,
                cudaStream_t s) {
  DeviceInfo di;
  if (int e = current_device_info(&di)) return e;
  shift_kernel<<<di.sm_count * 4, 256, 0, s>>>(off, adj, n_part, nnz_part, off_shift, id_shift);
  BFS_CUDA_TRY(cudaGetLastError());
  return BFS_OK;
}

int build_transpose(const int64_t* d_off, const int32_t* d_adj, int32_t n, int64_t nnz, cudaStream_t s,
                    int64_t** d_toff, int32_t** d_tadj) {
  DeviceInfo di;
  if (int e = current_device_info(&di)) return e;
  int32_t* src = nullptr;
  if (int e = dev_alloc((void**)&src, sizeof(int32_t) * (size_t)(nnz > 0 ? nnz : 1), "arc tails")) return e;
  expand_rows_kernel<<<di.sm_count * 8, 256, 0, s>>>(d_off, n, nnz, src);
  cudaError_t err = cudaGetLastError();
  if (err != cudaSuccess) {
    dev_free(src);
    return cuda_fail(err, "arc tails");
  }
  int64_t tnnz = 0;
  const int rc = build_csr_from_edges(src, d_adj, nnz, n, 2, s, d_toff, d_tadj, &tnnz);
  dev_free(src);
  if (rc) return rc;
  if (tnnz != nnz) {
    dev_free(*d_toff);
    dev_free(*d_tadj);
    return fail(BFS_ERR_INVALID_GRAPH, "transpose: the CSR has repeated arcs or self-loops");
  }
  return BFS_OK;
}

int check_offsets(const int64_t* d_off, int32_t n, int64_t nnz, int* d_flag, cudaStream_t s, int* ok) {
  DeviceInfo di;
  if (int e = current_device_info(&di)) return e;
  int bad = 0;
  cudaError_t err = cudaMemsetAsync(d_flag, 0, sizeof(int), s);
  if (err == cudaSuccess) {
    offsets_kernel<<<di.sm_count * 4, 256, 0, s>>>(d_off, n, nnz, d_flag);
    err = cudaGetLastError();
  }
  if (err == cudaSuccess) err = cudaMemcpyAsync(&bad, d_flag, sizeof(int), cudaMemcpyDeviceToHost, s);
  if (err == cudaSuccess) err = cudaStreamSynchronize(s);
  if (err != cudaSuccess) return cuda_fail(err, "row offset check");
  *ok = bad == 0;
  return BFS_OK;
}

int validate_csr(const int64_t* d_off, const int32_t* d_adj, int32_t n, int64_t nnz, bool symmetric, cudaStream_t s,
                 int* ok) {
  DeviceInfo di;
  if (int e = current_device_info(&di)) return e;
  int* d_bad = nullptr;
  if (int e = dev_alloc((void**)&d_bad, sizeof(int), "validation flag")) return e;
  int bad = 0;
  cudaError_t err = cudaMemsetAsync(d_bad, 0, sizeof(int), s);
  if (err == cudaSuccess) {
    validate_kernel<<<di.sm_count * 4, 256, 0, s>>>(d_off, d_adj, n, nnz, symmetric ? 1 : 0, d_bad);
    err = cudaGetLastError();
  }
  if (err == cudaSuccess) err = cudaMemcpyAsync(&bad, d_bad, sizeof(int), cudaMemcpyDeviceToHost, s);
  if (err == cudaSuccess) err = cudaStreamSynchronize(s);
  dev_free(d_bad);
  if (err != cudaSuccess) return cuda_fail(err, "CSR validation");
  *ok = bad == 0;
  return BFS_OK;
}

}  // namespace bfsint
