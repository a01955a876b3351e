// Level-synchronous BFS as one persistent cooperative kernel per traversal.
//
// Each level k is one sparse matrix-sparse vector product over the
// (select2nd, max) semiring followed by the mask with the visited set, the
// parent update and the frontier replacement (Sec. 3.2, Algorithm 3 on one
// device).  A level is one phase of the kernel; phases are separated by a
// grid-wide barrier, and the loop's control (frontier size, variant choice,
// termination) lives on the device, so a whole traversal is a single launch.
//
// State of a phase k (all in HBM, the bitmaps stay resident in L2):
//   cur  = bits[k % 3]        frontier f_k as a bitmap (read only)
//   nxt  = bits[(k + 1) % 3]  f_{k+1} being built (claims by atomicOr / owner stores)
//   clr  = bits[(k + 2) % 3]  f_{k-1}, cleared during the phase for reuse as nxt
//   vis  = visited bitmap; during phase k it holds levels <= k-1 (and possibly k),
//          so "reached" is tested as (vis | cur)
//   queue[k % 3]              f_k as a list; queue[(k + 1) % 3] receives f_{k+1}
//   ctr[k % 64]               counters of f_k (size, degree sum, degree bins)
//
// Variants (identical results):
//   top-down (thread / warp / degree-binned): for u in f_k and every neighbour w
//     not yet reached, atomicMax(parent[w], u) -- every frontier neighbour of w
//     contributes, so parent[w] ends as the largest-id one -- and the first
//     atomicOr on nxt claims w (level, queue, counters).  Frontier entries are
//     dealt round-robin over the CTAs so that small frontiers use every SM, and
//     vertices above the chunk degree are split into grid-wide chunk items of
//     kChunkEdges edges, one CTA each.
//   pull: for every vertex v not yet reached, scan its sorted row from the
//     largest id down; the first neighbour in f_k is the max-id parent.  One
//     warp owns a chunk of bitmap words at a time; the chunk's live rows are
//     dealt to the lanes, two per lane, and first tested against their probe
//     record (the row's largest ids); rows still open are collected per warp and
//     scanned one per lane.  Vertices without edges are marked
//     visited at init, so pull levels never touch them.
#include <cooperative_groups.h>
#include <cooperative_groups/scan.h>

#include <algorithm>
#include <mutex>
#include <climits>
#include <cstdio>
#include <type_traits>

#include "device_common.cuh"
#include "internal.h"
#include "claims.cuh"
#include "mlp_device.cuh"

namespace cg = cooperative_groups;

namespace bfsint {
namespace {

using bfsdev::kFull;

constexpr int kBlock = 512;
constexpr int kWarps = kBlock / 32;

#ifdef BFS_PHASE_TIMING
// Diagnostic build only: global-timer stamps of the first 4096 levels.
// [0] CTA 0 at level start, [1] after recycling, [2] after selection,
// [3] after expansion, [4] after counter flush, [5] latest barrier arrival
// of any CTA, [6] CTA 0 after the barrier.
__device__ unsigned long long g_phase_ts[4096][8];
#define PHASE_TS(k, slot)                                                             \
  do {                                                                                \
    if (blockIdx.x == 0 && threadIdx.x == 0 && (k) < 4096) g_phase_ts[k][slot] = bfsdev::global_timer_ns(); \
  } while (0)
#define PHASE_ARRIVAL(k)                                                              \
  do {                                                                                \
    __syncthreads();                                                                  \
    if (threadIdx.x == 0 && (k) < 4096) atomicMax(&g_phase_ts[k][5], (unsigned long long)bfsdev::global_timer_ns()); \
  } while (0)
#else
#define PHASE_TS(k, slot) \
  do {                    \
  } while (0)
#define PHASE_ARRIVAL(k) \
  do {                   \
  } while (0)
#endif

struct LoopParams {
  const int64_t* __restrict__ off;    // out-rows: top-down expansion
  const int32_t* __restrict__ adj;
  const int64_t* __restrict__ toff;   // in-rows: pull scans (the same arrays when undirected)
  const int32_t* __restrict__ tadj;
  int32_t directed;
  const uint32_t* __restrict__ dead;  // vertices no arc enters (and the tail), or null
  int32_t n;
  int32_t nwords;
  long long nnz;
  int32_t* level;
  int32_t* parent;
  int32_t* queue[3];
  uint32_t* bits[3];
  uint32_t* vis;
  int64_t* chunks[2];
  long long chunk_cap;  // entries of each chunk list
  LevelCtr* ctr;
  bfsdev::GridBarrier* bar;
  int* status;
  bfs_level_stat* stats;
  int32_t* misc;
  long long* edges_out;
  const int32_t* sources;  // device list when nsources > 1
  int32_t src0;            // the source when nsources == 1
  int32_t nsources;
  int32_t selector;
  int32_t forced;
  const int32_t* schedule;
  int32_t schedule_len;
  const float* mlp;
  float feat_log_n, feat_log_nnz, feat_inv_n, feat_inv_nnz;  // graph constants of the selector's features
  int32_t want_stats;
  unsigned spin_limit;
  int32_t warp_deg, cta_deg, pull_thread_deg, chunk_deg;
  float alpha, beta;
  long long small_frontier;  // TD_WARP for top-down levels up to this many vertices, all of degree <= 32
  long long narrow_edges;    // levels whose frontier has at most this many edges run on half the CTAs
  int32_t parts;
  const int64_t* part_base;
  int32_t** part_out;  // [2 * parts]: level outputs then parent outputs
  // 2D tiles of the in-adjacency for the tiled variant (t_jc null when absent)
  const uint16_t* __restrict__ t_jc;
  const uint32_t* __restrict__ t_cp;
  const uint16_t* __restrict__ t_ir;
  const int64_t* __restrict__ t_dir_jc;
  const int64_t* __restrict__ t_dir_ir;
  int32_t t_rb_bits, t_cb_bits, t_nrb, t_ncb;
  const int4* __restrict__ probe;  // per vertex an arc enters: in-degree and its row's largest three ids, or null
  const uint32_t* __restrict__ rank;  // per bitmap word: the records before it
  long long flat_visits;           // top-down: visits per thread up to which a small frontier's edges are dealt flat
  int32_t pull_words;              // bitmap words per pull chunk
  int32_t claim_by_parent;         // top-down: the first offer to a parent claims the vertex (else the next bitmap does)
  int32_t fr_shift;                // pull: log2 of the vertices per shared-memory frontier bit
  unsigned fr_limit;               // pull: largest frontier summarised in shared memory when fr_shift > 0
};

// Per-thread accumulation of the next frontier's counters.
struct Acc {
  unsigned long long edges = 0;
  unsigned b0 = 0, b1 = 0, b2 = 0;  // one thread claims fewer than 2^32 vertices
};

__device__ __forceinline__ void acc_vertex(Acc& a, long long deg) {
  a.edges += (unsigned long long)deg;
  if (deg <= 32) a.b0 += 1;
  else if (deg <= 1024) a.b1 += 1;
  else a.b2 += 1;
}

// Bookkeeping of a vertex claimed for level knext (the caller already set nxt).
__device__ __forceinline__ void claim_topdown(const LoopParams& p, int knext, int w, long long deg, Acc& acc,
                                              Claims& cl, int room) {
  p.level[w] = knext;
  cta_enqueue(p, knext, cl, w, room);
  acc_vertex(acc, deg);
  if (deg > p.chunk_deg) push_chunks_cta(p, knext, cl, w, deg);
}

// Top-down visits of up to N edges (u[i] -> w[i]) in phase k (w[i] < 0: none).
// Each kind of load is issued for all of them before any is used: a visit is a
// chain of three dependent round trips to L2 or DRAM.  room: see cta_enqueue.
template <int N>
__device__ __forceinline__ void td_visit(const LoopParams& p, const uint32_t* cur, uint32_t* nxt, int k,
                                         const int (&u)[N], const int (&w)[N], Acc& acc, Claims& cl, int room = kQBuf) {
  uint32_t reached[N], nw[N];
#pragma unroll
  for (int i = 0; i < N; ++i) {
    reached[i] = 0xffffffffu;
    nw[i] = 0;
    const bool live = bfsdev::kBoundsCheck ? u[i] >= 0 && bfsdev::in_range(p.status, bfsdev::kSiteTopDown, w[i], p.n) : u[i] >= 0;
    if (live) {
      const int ww = w[i] >> 5;
      reached[i] = p.vis[ww] | cur[ww];
      if (!p.claim_by_parent) nw[i] = nxt[ww];
    }
  }
  bool mine[N];
  long long deg[N];
#pragma unroll
  for (int i = 0; i < N; ++i) {
    const uint32_t m = 1u << (w[i] & 31);
    mine[i] = false;
    deg[i] = 0;
    if (reached[i] & m) continue;
    if (p.claim_by_parent) {
      // the offer itself tells who came first: parents of unreached vertices are -1
      deg[i] = __ldg(&p.off[w[i] + 1]) - __ldg(&p.off[w[i]]);  // speculative: the claim needs the degree
      mine[i] = atomicMax(&p.parent[w[i]], u[i]) < 0;
    } else {
      bfsdev::red_max_i32(&p.parent[w[i]], u[i]);
      if (nw[i] & m) continue;
      deg[i] = __ldg(&p.off[w[i] + 1]) - __ldg(&p.off[w[i]]);
      mine[i] = !(atomicOr(&nxt[w[i] >> 5], m) & m);
    }
  }
#pragma unroll
  for (int i = 0; i < N; ++i) {
    if (mine[i]) {
      if (p.claim_by_parent) atomicOr(&nxt[w[i] >> 5], 1u << (w[i] & 31));
      claim_topdown(p, k + 1, w[i], deg[i], acc, cl, room);
    }
  }
}

// One edge.
__device__ __forceinline__ void td_visit(const LoopParams& p, const uint32_t* cur, uint32_t* nxt, int k, int u, int w,
                                         Acc& acc, Claims& cl, int room = kQBuf) {
  const int u1[1] = {u}, w1[1] = {w};
  td_visit<1>(p, cur, nxt, k, u1, w1, acc, cl, room);
}

// 64-bit warp sum.
__device__ __forceinline__ unsigned long long warp_sum_u64(unsigned long long v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
  return v;
}

// End of a phase: the CTA's counter contributions, its buffered queue entries
// and its buffered chunk items go to level knext with one atomic each.  CTAs that
// claimed nothing skip all of it.  room: see cta_enqueue.
template <typename S>
__device__ __forceinline__ void end_phase(const LoopParams& p, int knext, Acc& acc, S& sm, int room = kQBuf) {
  const bool mine = (acc.b0 | acc.b1 | acc.b2) != 0;
  if (__syncthreads_or(mine)) {
    // n < 2^31 vertices in all: a warp's counts fit 32 bits
    const unsigned long long e = warp_sum_u64(acc.edges);
    const unsigned b0 = __reduce_add_sync(kFull, acc.b0), b1 = __reduce_add_sync(kFull, acc.b1),
                   b2 = __reduce_add_sync(kFull, acc.b2);
    if ((threadIdx.x & 31) == 0 && (e | b0 | b1 | b2)) {
      atomicAdd(&sm.acc[0], e);
      atomicAdd(&sm.acc[1], (unsigned long long)b0);
      atomicAdd(&sm.acc[2], (unsigned long long)b1);
      atomicAdd(&sm.acc[3], (unsigned long long)b2);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      LevelCtr* c = &p.ctr[knext % kCtrRing];
      if (sm.acc[0]) atomicAdd(&c->edges, sm.acc[0]);
      if (sm.acc[1]) atomicAdd(&c->bins[0], sm.acc[1]);
      if (sm.acc[2]) atomicAdd(&c->bins[1], sm.acc[2]);
      if (sm.acc[3]) atomicAdd(&c->bins[2], sm.acc[3]);
      sm.acc[0] = sm.acc[1] = sm.acc[2] = sm.acc[3] = 0;
    }
  }
  flush_claims(p, knext, sm.cl, room);
  acc = Acc{};
}

// The CTA's state.  With kLong the phases' area follows it in shared memory, behind the claim buffer.
struct __align__(64) Smem {
  float4 mlp_y;  // outputs of the selector network
  LevelCtr ctr;  // counters of the level to expand, fetched by thread 0 at the barrier before it
  int owner;
  int cu;
  long long cb, ce;
  int warp_tmp[kWarps + 1];
  unsigned long long acc[4];
  Claims cl;
};

// ---------------- top-down phase ----------------
// Dynamic shared memory of the top-down and tiled phases: frontier rows of a
// CTA with the prefix sums of their lengths.
constexpr int kFlatRows = 4 * kBlock;  // frontier vertices of a level whose edges are dealt to the whole grid
struct FlatSmem {
  long long tb[kFlatRows];
  int tu[kFlatRows];
  int tpref[kFlatRows + 1];
};

// The last of `rows` rows whose prefix sum is at most idx (a non-empty one when idx is below the total).
__device__ __forceinline__ int flat_owner(const FlatSmem& fl, int rows, int idx) {
  int lo = 0, hi = rows;
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (fl.tpref[mid] <= idx) lo = mid;
    else hi = mid;
  }
  return lo;
}

// Top-down level of a small frontier (at most kFlatRows vertices, few enough
// edges for the CTAs' claim buffers): every CTA takes in the whole frontier and
// the prefix sums of its degrees, and edge i goes to thread i of the grid, so
// that a level is one round of loads wherever its edges are.  By rows, the
// first levels of an R-MAT traversal (2 to 100 vertices with hundreds to
// thousands of edges each) ran on as many CTAs as they had rows or 1,024-edge
// chunks, two visits deep: 22 us at scale 16 for 7 rows, 30 us at scale 22 for
// 98.
__device__ void flat_phase(const LoopParams& p, int k, unsigned count, Smem& sm, FlatSmem& fl, Acc& acc, unsigned G) {
  const uint32_t* cur = p.bits[k % 3];
  uint32_t* nxt = p.bits[(k + 1) % 3];
  const int32_t* Q = p.queue[k % 3];
  const int tid = threadIdx.x, per = ((int)count + kBlock - 1) / kBlock, rows = per * kBlock;
  int u[4], deg[4], sum = 0;
  long long b[4];
#pragma unroll
  for (int r = 0; r < 4; ++r) u[r] = r < per && tid * per + r < (int)count ? Q[tid * per + r] : -1;
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    b[r] = u[r] >= 0 ? __ldg(&p.off[u[r]]) : 0;
    deg[r] = u[r] >= 0 ? (int)(__ldg(&p.off[u[r] + 1]) - b[r]) : 0;
    sum += deg[r];
  }
  int at = 0;
  const int total = block_exclusive_scan(sum, sm.warp_tmp, at);
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    if (r < per) {
      fl.tu[tid * per + r] = u[r];
      fl.tb[tid * per + r] = b[r];
      fl.tpref[tid * per + r] = at;
      at += deg[r];
      if (u[r] >= 0 && (unsigned)(tid * per + r) % G == blockIdx.x) atomicOr(&p.vis[u[r] >> 5], 1u << (u[r] & 31));
    }
  }
  __syncthreads();
  int room = kQBuf / kBlock;  // steps that the CTA's claim buffer is sure to hold
  for (int base = (int)blockIdx.x * kBlock; base < total; base += (int)G * kBlock) {
    if (room-- == 0) {
      flush_claims_if_full(p, k + 1, sm.cl, kBlock, kBigBuf / 2);
      room = 0;
    }
    const int idx = base + tid;
    if (idx < total) {
      const int o = flat_owner(fl, rows, idx);
      td_visit(p, cur, nxt, k, fl.tu[o], __ldg(&p.adj[fl.tb[o] + (idx - fl.tpref[o])]), acc, sm.cl);
    }
  }
}

// A frontier row fetched ahead of the phase (u < 0: none).
struct FirstRow {
  int u = -1;
  long long b = 0, e = 0;
};

// kLong: the claim buffer of the thread and warp variants goes on into the phases'
// area, which they leave free: without a barrier in their loops, which a row of
// 1,024 edges would hold up, they cannot empty it on the way.
constexpr int kLongQ = 15040;  // entries (checked below)
template <bool kLong>
__device__ __forceinline__ int claim_room(int variant) {
  return kLong && (variant == BFS_VARIANT_TD_THREAD || variant == BFS_VARIANT_TD_WARP) ? kLongQ : kQBuf;
}

template <bool kLong>
__device__ void topdown_phase(const LoopParams& p, int k, int variant, unsigned count, unsigned nchunks,
                              const FirstRow& first, Smem& sm, FlatSmem& fl, Acc& acc, unsigned G) {
  const uint32_t* cur = p.bits[k % 3];
  uint32_t* nxt = p.bits[(k + 1) % 3];
  const int32_t* Q = p.queue[k % 3];
  const int tid = threadIdx.x, lane = tid & 31;
  constexpr int kRoom = kLong ? kLongQ : kQBuf;  // of the thread and warp variants

  // chunk items of high-degree frontier vertices: one CTA per item; before each
  // item the CTA makes room in its buffers for the item's claims
  const int64_t* items = p.chunks[k & 1];
  for (unsigned ci = blockIdx.x; ci < nchunks; ci += G) {
    flush_claims_if_full(p, k + 1, sm.cl, kChunkEdges, kBigBuf / 2);
    const int64_t it = items[ci];
    const int v = (int)(it >> 32);
    const long long c = it & 0xffffffffll;
    const long long rb = __ldg(&p.off[v]), re = __ldg(&p.off[v + 1]);
    const long long b = rb + c * kChunkEdges;
    const long long e = min(b + (long long)kChunkEdges, re);
    static_assert(kChunkEdges == 2 * kBlock, "two visits per thread and chunk");
    const int us[2] = {b + tid < e ? v : -1, b + kBlock + tid < e ? v : -1};
    const int ws[2] = {us[0] >= 0 ? __ldg(&p.adj[b + tid]) : 0, us[1] >= 0 ? __ldg(&p.adj[b + kBlock + tid]) : 0};
    td_visit<2>(p, cur, nxt, k, us, ws, acc, sm.cl);
  }
  // the items' claims, for which there was room in kQBuf, come before any claim past it
  if (kLong && nchunks) __syncthreads();

  // frontier entry i goes to CTA i % G, so that small frontiers spread over the SMs
  const long long gthreads = (long long)G * kBlock;
  if (variant == BFS_VARIANT_TD_THREAD) {
    for (long long i = blockIdx.x + (long long)tid * G; i < count; i += gthreads) {
      const int u = Q[i];
      atomicOr(&p.vis[u >> 5], 1u << (u & 31));
      const long long b = __ldg(&p.off[u]), e = __ldg(&p.off[u + 1]);
      if (e - b > p.chunk_deg) continue;
      for (long long j = b; j < e; ++j) td_visit(p, cur, nxt, k, u, __ldg(&p.adj[j]), acc, sm.cl, kRoom);
    }
  } else if (variant == BFS_VARIANT_TD_WARP) {
    const long long gwarps = gthreads / 32;
    FirstRow row = first;  // the row of entry blockIdx.x + warp * G, where it was fetched
    for (long long i = blockIdx.x + (long long)(tid >> 5) * G; i < count; i += gwarps) {
      if (row.u < 0) {
        row.u = Q[i];
        row.b = __ldg(&p.off[row.u]);
        row.e = __ldg(&p.off[row.u + 1]);
      }
      if (lane == 0) atomicOr(&p.vis[row.u >> 5], 1u << (row.u & 31));
      if (row.e - row.b <= p.chunk_deg)
        for (long long j = row.b + lane; j < row.e; j += 32)
          td_visit(p, cur, nxt, k, row.u, __ldg(&p.adj[j]), acc, sm.cl, kRoom);
      row.u = -1;
    }
  } else {  // BFS_VARIANT_TD_BINNED
    for (long long tile = 0; tile < count; tile += gthreads) {
      flush_claims_if_full(p, k + 1, sm.cl, kQBuf / 2, kBigBuf / 2);
      const long long i = tile + blockIdx.x + (long long)tid * G;
      int u = -1;
      long long b = 0, e = 0;
      if (i < count) {
        u = Q[i];
        atomicOr(&p.vis[u >> 5], 1u << (u & 31));
        b = __ldg(&p.off[u]);
        e = __ldg(&p.off[u + 1]);
        if (e - b > p.chunk_deg) u = -1;
      }
      const long long deg = u >= 0 ? e - b : 0;
      // CTA bin: the whole CTA walks one row at a time
      for (;;) {
        if (u >= 0 && deg >= p.cta_deg) sm.owner = tid;
        __syncthreads();
        const int owner = sm.owner;
        if (owner < 0) break;
        if (tid == owner) {
          sm.cu = u;
          sm.cb = b;
          sm.ce = e;
          u = -1;
        }
        __syncthreads();
        const int cu = sm.cu;
        const long long cb = sm.cb, ce = sm.ce;
        for (long long j = cb + tid; j < ce; j += kBlock) td_visit(p, cur, nxt, k, cu, __ldg(&p.adj[j]), acc, sm.cl);
        __syncthreads();
        if (tid == 0) sm.owner = -1;
        __syncthreads();
      }
      // warp bin: a warp walks one row at a time
      for (;;) {
        const unsigned wm = __ballot_sync(kFull, u >= 0 && deg >= p.warp_deg);
        if (!wm) break;
        const int l = __ffs(wm) - 1;
        const int cu = __shfl_sync(kFull, u, l);
        const long long cb = __shfl_sync(kFull, b, l), ce = __shfl_sync(kFull, e, l);
        if (lane == l) u = -1;
        for (long long j = cb + lane; j < ce; j += 32) td_visit(p, cur, nxt, k, cu, __ldg(&p.adj[j]), acc, sm.cl);
      }
      // thread bin: the CTA gathers the remaining short rows edge by edge
      const int sdeg = u >= 0 ? (int)deg : 0;
      int excl = 0;
      const int total = block_exclusive_scan(sdeg, sm.warp_tmp, excl);
      fl.tu[tid] = u;
      fl.tb[tid] = b;
      fl.tpref[tid] = excl;
      if (tid == 0) fl.tpref[kBlock] = total;
      __syncthreads();
      for (int base = 0; base < total; base += kBlock) {
        const int idx = base + tid;
        if (idx < total) {
          const int lo = flat_owner(fl, kBlock, idx);
          td_visit(p, cur, nxt, k, fl.tu[lo], __ldg(&p.adj[fl.tb[lo] + (idx - fl.tpref[lo])]), acc, sm.cl);
        }
      }
      __syncthreads();
    }
  }
}

// ---------------- pull phase ----------------
constexpr int kPullRows = 2;       // live rows per lane in flight
constexpr int kPullProbes = 3;     // top entries of a row tested from its probe record
constexpr int kFrWords = 2048;     // frontier test in shared memory: 65,536 bits.  8,192 words left the top-down
                                   // levels' bitmap loads too little L1 (77 K-vertex level: 37 -> 63 us)
static_assert(kPullProbes == 3, "the unpacking of the probe records below");
constexpr int kDefer = 112;        // deferred rows a warp can hold; scanned once fewer than 64 more would fit
constexpr int kScanRefill = 24;    // a deferred scan with this many open rows or fewer takes new ones
constexpr int kScanOpen = 8;       // a deferred scan with fewer open rows and none left to take hands them back
constexpr int kWarpRow = 128;      // remaining entries from which a row left open is scanned by the whole warp

// Dynamic shared memory of the pull phase.
struct __align__(16) PullSmem {
  uint32_t fr[kFrWords];
  uint32_t hits[kWarps][32];   // hit bits of each warp's bitmap words
  uint2 entry[kWarps][32];     // of each warp's bitmap words: the vertices with a record, the records before
  int4 defer[kWarps][kDefer];  // rows still open after their probe: vertex, entries not yet examined, row start (64 bits)
};

__device__ __forceinline__ unsigned smem_addr(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }

// Position of the r-th (0-based) set bit of m; r < popc(m).
__device__ __forceinline__ int select_bit(uint32_t m, int r) {
  int pos = 0;
#pragma unroll
  for (int s = 16; s >= 1; s >>= 1) {
    const int c = __popc(m & ((1u << s) - 1u));  // set bits in the low s bits
    if (r >= c) {
      r -= c;
      m >>= s;
      pos += s;
    }
  }
  return pos;
}

// The idx-th live vertex of a warp's chunk of bitmap words that starts at word
// w0 (all lanes call it; lane l holds word l's live bits `live` and the
// inclusive prefix `incl` of their counts).  Returns the vertex, the owner lane
// of its word and its bit.
__device__ __forceinline__ int live_vertex(int w0, uint32_t live, int incl, int idx, int& owner, uint32_t& bit) {
  int o = 0;  // number of lanes whose inclusive prefix is <= idx: the owner
#pragma unroll
  for (int st = 16; st >= 1; st >>= 1) {
    const int c = __shfl_sync(kFull, incl, o + st - 1);
    if (c <= idx) o += st;
  }
  o = min(o, 31);
  const uint32_t lo = __shfl_sync(kFull, live, o);
  const int excl_o = __shfl_sync(kFull, incl, o) - __popc(lo);
  const int b = select_bit(lo, max(idx - excl_o, 0));
  owner = o;
  bit = 1u << b;
  return (w0 + o) * 32 + b;
}

// Where a pull level tests "is u in f_k".
enum FrontierMode : int {
  kFrGlobal = 0,   // the bitmap in global memory (L2)
  kFrExact = 1,    // a copy of the whole bitmap in shared memory (n <= 32 * kFrWords)
  kFrSummary = 2,  // shared memory holds one bit per 2^fr_shift vertices; a set one is confirmed in the bitmap
};

struct FrontierTest {
  const uint32_t* cur;
  const uint32_t* fr;
  int shift;
  FrontierMode mode;
};

// Which of the N ids u (those with their bit in `valid`) are in f_k, as a bit
// mask; the loads of one call are in flight together.
template <int N>
__device__ __forceinline__ unsigned in_frontier(const LoopParams& p, const FrontierTest& f, const int (&u)[N],
                                                unsigned valid) {
  if constexpr (bfsdev::kBoundsCheck) {
#pragma unroll
    for (int q = 0; q < N; ++q)
      if (((valid >> q) & 1u) && !bfsdev::in_range(p.status, bfsdev::kSitePull, u[q], p.n)) valid &= ~(1u << q);
  }
  unsigned m = valid;
  if (f.mode != kFrGlobal) {
#pragma unroll
    for (int q = 0; q < N; ++q) {
      const unsigned y = (unsigned)u[q] >> f.shift;
      const unsigned t = (f.fr[(y >> 5) & (kFrWords - 1)] >> (y & 31)) & 1u;
      m &= ~((t ^ 1u) << q);
    }
    if (f.mode == kFrExact) return m;
  }
  uint32_t x[N];
#pragma unroll
  for (int q = 0; q < N; ++q) x[q] = ((m >> q) & 1u) ? f.cur[u[q] >> 5] : 0u;
  unsigned h = 0;
#pragma unroll
  for (int q = 0; q < N; ++q) h |= ((x[q] >> (u[q] & 31)) & 1u) << q;
  return h;
}

// Four consecutive entries of the in-adjacency from index i, which is a
// multiple of four entries from a 16-byte boundary; entries outside the array
// read as 0.
__device__ __forceinline__ int4 load_entries4(const LoopParams& p, long long i) {
  if (i >= 0 && i + 4 <= p.nnz) return __ldg(reinterpret_cast<const int4*>(p.tadj + i));
  int4 r = make_int4(0, 0, 0, 0);
  if (i >= 0 && i < p.nnz) r.x = __ldg(p.tadj + i);
  if (i + 1 >= 0 && i + 1 < p.nnz) r.y = __ldg(p.tadj + i + 1);
  if (i + 2 >= 0 && i + 2 < p.nnz) r.z = __ldg(p.tadj + i + 2);
  if (i + 3 >= 0 && i + 3 < p.nnz) r.w = __ldg(p.tadj + i + 3);
  return r;
}

// Start of the aligned group of four entries that holds entry i.
__device__ __forceinline__ long long group_start(const LoopParams& p, long long i) {
  const int a = (int)((reinterpret_cast<uintptr_t>(p.tadj) >> 2) & 3u);
  return ((i + a) & ~3ll) - a;
}

// The whole warp scans entries [b, t) of one row from the top, 128 per step;
// returns the first frontier neighbour (the largest id) or -1.
__device__ __forceinline__ int scan_row_warp(const LoopParams& p, const FrontierTest& f, long long b, long long t,
                                             int lane) {
  while (t > b) {
    const long long top = group_start(p, t - 1), g = top - 4 * lane;
    int u[4] = {0, 0, 0, 0};
    unsigned valid = 0;
    if (g + 3 >= b) {
      const int4 e = load_entries4(p, g);
      u[0] = e.w, u[1] = e.z, u[2] = e.y, u[3] = e.x;
#pragma unroll
      for (int q = 0; q < 4; ++q) valid |= (g + 3 - q >= b && g + 3 - q < t) ? 1u << q : 0u;
    }
    const unsigned h = in_frontier<4>(p, f, u, valid);
    const unsigned any = __ballot_sync(kFull, h != 0);
    if (any) {
      const int q = __ffs(h) - 1;
      const int mine = q == 0 ? u[0] : q == 1 ? u[1] : q == 2 ? u[2] : u[3];
      return __shfl_sync(kFull, mine, __ffs(any) - 1);
    }
    t = top - 124;
  }
  return -1;
}

// Bookkeeping of vertices reached by the pull (one per lane where hit >= 0, its
// parent): outputs, counters, chunk items and the warp's queue buffer.  deg_in
// is the in-degree.
__device__ __forceinline__ void pull_claim(const LoopParams& p, int knext, int v, int hit, long long deg_in, Acc& acc,
                                           Claims& cl, int* wq, int& nbuf, int lane) {
  if (hit >= 0) {
    p.parent[v] = hit;
    p.level[v] = knext;
    // out-degree: the next level expands v's out-row (the row scanned here when undirected)
    const long long deg = p.directed ? __ldg(&p.off[v + 1]) - __ldg(&p.off[v]) : deg_in;
    acc_vertex(acc, deg);
    if (deg > p.chunk_deg) push_chunks_cta(p, knext, cl, v, deg);
  }
  warp_enqueue(p, knext, wq, nbuf, hit >= 0, v, lane, false);
}

// Scans the warp's deferred rows, one per lane: eight entries (two aligned
// 16-byte loads) per step and row, from the top.  A lane whose row is done
// takes the next of the list, so that the lanes stay busy however different
// the rows' lengths are.  Once the list is empty and fewer than kScanOpen rows
// are open, those go back to the list (with `flush`: are scanned to their
// end), except that one with kWarpRow or more entries left is scanned by the
// whole warp.
__device__ __forceinline__ void scan_deferred(const LoopParams& p, const FrontierTest& f, int knext, uint32_t* nxt,
                                              int4* defer, int& nd, bool flush, Acc& acc, Claims& cl, int* wq,
                                              int& nbuf, int lane) {
  asm volatile("cp.async.wait_all;" ::: "memory");  // the row starts of the list
  __syncwarp();
  int v = -1, hit = -1;
  long long b = 0, t = 0;
  bool open = false;
  for (;;) {
    unsigned m = __ballot_sync(kFull, open);
    if (__popc(m) <= kScanRefill) {
      if (nd == 0 && __popc(m) < kScanOpen) {
        for (unsigned big = __ballot_sync(kFull, open && t - b >= kWarpRow); big; big &= big - 1u) {
          const int l = __ffs(big) - 1;
          const int r = scan_row_warp(p, f, __shfl_sync(kFull, b, l), __shfl_sync(kFull, t, l), lane);
          if (lane == l) {
            hit = r;
            open = false;
          }
        }
      }
      if (__any_sync(kFull, hit >= 0)) {
        long long deg = 0;
        if (hit >= 0) {
          atomicOr(&nxt[v >> 5], 1u << (v & 31));
          if (!p.directed) deg = __ldg(&p.toff[v + 1]) - b;
        }
        pull_claim(p, knext, v, hit, deg, acc, cl, wq, nbuf, lane);
        hit = -1;
      }
      m = __ballot_sync(kFull, open);
      if (nd > 0) {
        const int i = nd - 1 - __popc(~m & bfsdev::lanemask_lt());
        if (!open && i >= 0) {
          const int4 d = defer[i];
          v = d.x;
          b = (long long)(((unsigned long long)(unsigned)d.w << 32) | (unsigned)d.z);
          t = b + d.y;
          open = true;
        }
        nd = max(0, nd - __popc(~m));
      } else if (m == 0) {
        break;
      } else if (!flush && __popc(m) < kScanOpen) {
        __syncwarp();  // every lane has read its entry
        if (open)
          defer[__popc(m & bfsdev::lanemask_lt())] = make_int4(v, (int)(t - b), (int)b, (int)(b >> 32));
        nd = __popc(m);
        break;
      }
    }
    if (open) {
      const long long g1 = group_start(p, t - 1), g0 = g1 - 4;
      const int4 e1 = load_entries4(p, g1);
      int4 e0 = make_int4(0, 0, 0, 0);
      if (g1 > b) e0 = load_entries4(p, g0);
      const int u[8] = {e1.w, e1.z, e1.y, e1.x, e0.w, e0.z, e0.y, e0.x};
      const int skip = (int)(g1 + 4 - t);  // entries of the top group at or above t
      const int cnt = (int)min((long long)(8 - skip), t - b);
      const unsigned h = in_frontier<8>(p, f, u, ((1u << cnt) - 1u) << skip);
      if (h) {
        const unsigned first = h & (0u - h);
#pragma unroll
        for (int q = 0; q < 8; ++q)
          if (first == 1u << q) hit = u[q];
        open = false;
      } else {
        t -= cnt;
        open = t > b;
      }
    }
  }
  __syncwarp();
}

// Dense-frontier SpMV over the unvisited rows.  A warp takes a chunk of
// pull_words bitmap words (32 vertices each) at a time: lane l loads word l of
// `vis` and of `cur`, and the chunk's live vertices (not reached, not
// edgeless) are dealt to the lanes 64 at a time, two rows per lane, so that
// every lane carries a row however sparse the live vertices are.
//
// The top entries of a row come from its probe record (degree and largest
// three ids, 16 bytes per vertex that an arc enters, built with the graph): on an R-MAT graph's
// dense level nearly every row ends there, and the records of a chunk are
// read in order, where the rows' own ends are one DRAM sector each at random.
// Rows still open go to a list of the warp, their starts fetched into it with
// cp.async; once it fills, they are scanned one per lane, eight entries per
// step (scan_deferred), so that a warp has 256 entries in flight instead of
// the 32 of a scan that packs the open rows into one load per lane.
//
// The frontier test reads shared memory where it can: an exact copy of the
// bitmap up to 65,536 vertices, and above that, for a frontier of at most
// fr_limit vertices, one bit per 2^fr_shift vertices, which rejects all but a
// few percent of the entries (the first pull level of a traversal led by hubs
// tests half a billion entries at scale 26 against a few thousand vertices).
//
// Chunk size and deal: a chunk costs its warp about 3.5 us of dependent loads
// however few live rows it holds, so a graph of up to 32 words per resident
// warp gives every warp one chunk (32-word chunks for all sizes left 64 of
// 4,864 warps with work at scale 16), and larger graphs use 32-word chunks.
// Rows without a frontier neighbour near their top make some chunks far dearer
// than others, so the second half of a large level's chunks is handed out
// dynamically (with an all-dynamic deal the cursor's atomics, all at once at
// the start of a level, cost more than they save).
//
// What bounds it: the latency of the chain bitmap words -> record -> frontier
// test -> row, with 8 warps per scheduler to hide it, and on a dense level
// at scale 26 DRAM (records, outputs written over their -1 fill).  Measured
// against a pull that read the rows' bounds and top entries and packed the open
// rows into one load per lane (level times, R-MAT edgefactor 16): scale 26, f_k
// of 5,328 vertices 2,341 -> 1,270 us, of 9.6 M 615 -> 373 us, of 2.9 M 713 ->
// 455 us; scale 22, f_k of 3,946 vertices 162 -> 80 us; scale 16, f_k of 4,525
// vertices 33 -> 13 us.
__device__ void pull_phase(const LoopParams& p, int k, unsigned count, Smem& sm, PullSmem& ps, Acc& acc, unsigned G) {
  uint32_t* nxt = p.bits[(k + 1) % 3];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const long long gwarps = (long long)G * kWarps;
  const int knext = k + 1;
  const int probe = min(p.pull_thread_deg, kPullProbes);  // the tuning knob, at most kPullProbes
  FrontierTest f{p.bits[k % 3], ps.fr, p.fr_shift, kFrGlobal};
  if (p.fr_shift == 0) {
    f.mode = kFrExact;
    for (int i = threadIdx.x; i < p.nwords; i += kBlock) ps.fr[i] = f.cur[i];
    __syncthreads();
  } else if (count <= p.fr_limit) {
    f.mode = kFrSummary;
    for (int i = threadIdx.x; i < kFrWords / 4; i += kBlock) reinterpret_cast<uint4*>(ps.fr)[i] = make_uint4(0, 0, 0, 0);
    __syncthreads();
    const int32_t* Q = p.queue[k % 3];
#pragma unroll 4
    for (unsigned i = threadIdx.x; i < count; i += kBlock) {
      const unsigned y = (unsigned)Q[i] >> p.fr_shift;
      atomicOr(&ps.fr[(y >> 5) & (kFrWords - 1)], 1u << (y & 31));
    }
    __syncthreads();
  }
  int* wq = sm.cl.wq[wid];
  uint32_t* hitw = ps.hits[wid];
  uint2* entry = ps.entry[wid];
  int4* defer = ps.defer[wid];
  int nbuf = 0, nd = 0;
  // chunk indices fit 32 bits: nwords < 2^26
  const int W = p.pull_words, nchunks = (p.nwords + W - 1) / W, gw = (int)gwarps;
  // Chunks [0, S) are dealt statically (warp i takes i, i + gw, ...), the
  // rest from the level's cursor, each fetch issued one chunk ahead.  With
  // fewer than two chunks per warp the level is all static (S past every chunk).
  const int S = nchunks > 2 * gw ? gw * max(1, (nchunks / 2) / gw) : INT_MAX;
  for (int c = wid * (int)G + (int)blockIdx.x;;) {
    const bool more = c < nchunks;  // after the last chunk one more turn scans what is left deferred
    unsigned taken = 0;
    if (more && c + gw >= S && lane == 0) taken = (unsigned)atomicAdd(&p.ctr[k % kCtrRing].pad, 1ull);  // used after the chunk
    const int w0 = c * W, w = w0 + lane;
    const bool has = more && lane < W && w < p.nwords;
    const uint32_t vw = has ? p.vis[w] : 0xffffffffu;
    const uint32_t cw = has ? f.cur[w] : 0u;
    const uint32_t visw = vw | cw;
    const uint32_t live = ~visw;
    if (p.probe != nullptr && has) entry[lane] = make_uint2(~__ldg(&p.dead[w]), __ldg(&p.rank[w]));
    const int cnt = __popc(live);
    int incl = cnt;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(kFull, incl, o);
      if (lane >= o) incl += y;
    }
    const int total = __shfl_sync(kFull, incl, 31);
    hitw[lane] = 0u;
    __syncwarp();
    for (int base = 0;; base += 32 * kPullRows) {
      if (nd > kDefer - 32 * kPullRows || !more)
        scan_deferred(p, f, knext, nxt, defer, nd, !more, acc, sm.cl, wq, nbuf, lane);
      if (base >= total) break;
      int v[kPullRows], o[kPullRows], deg[kPullRows], u[kPullRows * kPullProbes];
      uint32_t bit[kPullRows];
#pragma unroll
      for (int r = 0; r < kPullRows; ++r) {
        const int i = base + r * 32 + lane;
        const int lv = live_vertex(w0, live, incl, min(i, total - 1), o[r], bit[r]);
        v[r] = i < total ? lv : -1;
      }
      if (p.probe != nullptr) {
#pragma unroll
        for (int r = 0; r < kPullRows; ++r) {
          const uint2 en = entry[o[r]];
          const uint32_t at = en.y + __popc(en.x & (bit[r] - 1u));
          const int4 rec = v[r] >= 0 ? __ldg(&p.probe[at]) : make_int4(0, 0, 0, 0);
          deg[r] = rec.x;
          u[3 * r] = rec.y, u[3 * r + 1] = rec.z, u[3 * r + 2] = rec.w;
        }
      } else {  // no records (the static entry point): the same from the row itself
#pragma unroll
        for (int r = 0; r < kPullRows; ++r) {
          const long long b = v[r] >= 0 ? __ldg(&p.toff[v[r]]) : 0, e = v[r] >= 0 ? __ldg(&p.toff[v[r] + 1]) : 0;
          deg[r] = (int)(e - b);
#pragma unroll
          for (int q = 0; q < kPullProbes; ++q) u[3 * r + q] = q < deg[r] ? __ldg(&p.tadj[e - 1 - q]) : 0;
        }
      }
      unsigned valid = 0;  // one test of both rows: all its loads are in flight together
#pragma unroll
      for (int r = 0; r < kPullRows; ++r) valid |= ((1u << min(probe, deg[r])) - 1u) << (3 * r);
      const unsigned found = in_frontier<kPullRows * kPullProbes>(p, f, u, valid);
#pragma unroll
      for (int r = 0; r < kPullRows; ++r) {
        const unsigned h = found >> (3 * r) & 7u;
        const int hit = h == 0 ? -1 : (h & 1u) ? u[3 * r] : (h & 2u) ? u[3 * r + 1] : u[3 * r + 2];
        const bool later = hit < 0 && deg[r] > probe;
        const unsigned m = __ballot_sync(kFull, later);
        if (later) {
          int4* d = &defer[nd + __popc(m & bfsdev::lanemask_lt())];
          *reinterpret_cast<int2*>(d) = make_int2(v[r], deg[r] - probe);
          asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(smem_addr(d) + 8), "l"(p.toff + v[r]) : "memory");
        }
        nd += __popc(m);
        if (hit >= 0) atomicOr(&hitw[o[r]], bit[r]);
        pull_claim(p, knext, v[r], hit, deg[r], acc, sm.cl, wq, nbuf, lane);
      }
      __syncwarp();
    }
    if (!more) break;
    const uint32_t hits = hitw[lane];
    if (has) {
      // the deferred rows of this word OR their hits in as they are found; the
      // next level's pull folds nxt into vis, so vis need not hold them yet
      if (hits) atomicOr(&nxt[w], hits);
      if ((visw | hits) != vw) p.vis[w] = visw | hits;
    }
    __syncwarp();
    c = c + gw >= S ? S + (int)__shfl_sync(kFull, taken, 0) : c + gw;
  }
  warp_enqueue(p, knext, wq, nbuf, false, 0, lane, true);
}

// ---------------- tiled phase ----------------
// Dense-frontier SpMV over the 2D tiles of the in-adjacency (Sec. 3.2's 2D
// blocks, each in the DCSC form of Sec. 4.1).  A CTA owns a row block at a
// time and keeps two tile-local slices in shared memory: `done`, the row
// block's reached rows (vis | cur at level start, plus the rows found in the
// tiles already walked), and `slice`, the frontier bits of the current column
// block.  It walks the row block's tiles from the highest column block down;
// in each tile the non-empty columns that are in the frontier expand their
// rows (flattened over the CTA by a prefix sum, like the thread bin of the
// top-down phase), and every row not yet done takes the column as a parent
// candidate with atomicMax.  A row's candidates all come from the first tile
// (in that order) that holds a frontier neighbour, since `done` only changes
// between tiles, so the largest candidate is its max-id parent.  The row
// block's found rows then go out as in the pull: owner-written nxt / vis
// words, levels, counters and the warp queue buffers.
constexpr int kTileWordsMax = 2048;  // 2^16 rows or columns per tile

__device__ void tiled_phase(const LoopParams& p, int k, Smem& sm, FlatSmem& fl, uint32_t* tsm, Acc& acc,
                            unsigned G) {
  const uint32_t* cur = p.bits[k % 3];
  uint32_t* nxt = p.bits[(k + 1) % 3];
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const int knext = k + 1;
  uint32_t* done = tsm;
  uint32_t* newf = tsm + kTileWordsMax;
  uint32_t* slice = tsm + 2 * kTileWordsMax;
  const int rbw = 1 << (p.t_rb_bits - 5), cbw = 1 << (p.t_cb_bits - 5);
  int* wq = sm.cl.wq[wid];
  int nbuf = 0;
  for (int rb = blockIdx.x; rb < p.t_nrb; rb += G) {
    const long long w0 = (long long)rb * rbw;
    bool live = false;
    for (int i = tid; i < rbw; i += kBlock) {
      const long long w = w0 + i;
      const uint32_t d = w < p.nwords ? (p.vis[w] | cur[w]) : 0xffffffffu;
      done[i] = d;
      newf[i] = 0u;
      live |= d != 0xffffffffu;
    }
    // a block whose rows are all reached walks no tile, but still folds cur into vis below
    const int first_cb = __syncthreads_or(live) ? p.t_ncb - 1 : -1;
    for (int cb = first_cb; cb >= 0; --cb) {
      const long long t = (long long)rb * p.t_ncb + cb;
      const long long j0 = p.t_dir_jc[t], j1 = p.t_dir_jc[t + 1];
      if (j0 == j1) continue;  // empty tile (the same on every thread)
      const long long ibase = p.t_dir_ir[t], iend = p.t_dir_ir[t + 1];
      const long long s0 = (long long)cb * cbw;
      for (int i = tid; i < cbw; i += kBlock) slice[i] = s0 + i < p.nwords ? cur[s0 + i] : 0u;
      __syncthreads();
      bool tile_hit = false;
      for (long long jb = j0; jb < j1; jb += kBlock) {
        const long long j = jb + tid;
        int ul = -1;
        long long rbeg = 0, rlen = 0;
        if (j < j1) {
          const int c = p.t_jc[j];
          if ((slice[c >> 5] >> (c & 31)) & 1u) {
            ul = c;
            rbeg = ibase + p.t_cp[j];
            rlen = (j + 1 < j1 ? ibase + p.t_cp[j + 1] : iend) - rbeg;
          }
        }
        int excl = 0;
        const int total = block_exclusive_scan((int)rlen, sm.warp_tmp, excl);
        fl.tu[tid] = ul;
        fl.tb[tid] = rbeg;
        fl.tpref[tid] = excl;
        if (tid == 0) fl.tpref[kBlock] = total;
        __syncthreads();
        for (int base = 0; base < total; base += kBlock) {
          const int idx = base + tid;
          if (idx < total) {
            const int lo = flat_owner(fl, kBlock, idx);  // a frontier column with rows
            const int r = p.t_ir[fl.tb[lo] + (idx - fl.tpref[lo])];
            if (!((done[r >> 5] >> (r & 31)) & 1u)) {
              atomicMax(&p.parent[(rb << p.t_rb_bits) + r], (cb << p.t_cb_bits) + fl.tu[lo]);
              atomicOr(&newf[r >> 5], 1u << (r & 31));
              tile_hit = true;
            }
          }
        }
        __syncthreads();
      }
      // the tile's rows are done from here on; stop once every row of the block is
      if (__syncthreads_or(tile_hit)) {
        live = false;
        for (int i = tid; i < rbw; i += kBlock) {
          const uint32_t d = done[i] | newf[i];
          done[i] = d;
          newf[i] = 0u;
          live |= d != 0xffffffffu;
        }
        if (!__syncthreads_or(live)) break;
      }
    }
    // rows found in this row block: done now minus reached at level start; every
    // word of the block gets vis |= cur | found, as in the pull phase, so that
    // f_k stays reached after its bitmap is recycled
    for (int i = wid; i < rbw; i += kWarps) {
      const long long w = w0 + i;
      if (w >= p.nwords) break;
      const uint32_t vw = p.vis[w], cw = cur[w];
      const uint32_t visw = vw | cw;
      const uint32_t f = done[i] & ~visw;
      if (lane == 0) {
        if (f) nxt[w] = f;
        if ((visw | f) != vw) p.vis[w] = visw | f;
      }
      const bool hit = (f >> lane) & 1u;
      const int v = (int)(w * 32 + lane);
      if (hit) {
        p.level[v] = knext;
        const long long deg = __ldg(&p.off[v + 1]) - __ldg(&p.off[v]);
        acc_vertex(acc, deg);
        if (deg > p.chunk_deg) push_chunks_cta(p, knext, sm.cl, v, deg);
      }
      warp_enqueue(p, knext, wq, nbuf, hit, v, lane, false);
    }
    __syncthreads();
  }
  warp_enqueue(p, knext, wq, nbuf, false, 0, lane, true);
}

// The selector network on four warps of the CTA (tid counts from their first),
// on the parameters in the warp layout; its outputs go to y.
__device__ __forceinline__ void learned_outputs(const LoopParams& p, const float* w, bfsdev::MlpScratch& sc, float* y,
                                             int tid, int k, const LevelCtr& c, long long unvisited,
                                             long long unvisited_edges) {
  float x[12];
  bfsdev::warp_level_features(p.feat_log_n, p.feat_log_nnz, p.feat_inv_n, p.feat_inv_nnz, k, c.count,
                              (long long)c.edges, unvisited, unvisited_edges, c.bins, tid & 31, x);
  bfsdev::warps_mlp_outputs(w, x, sc, y, tid >> 5, tid & 31);
}

// Direction choice in the manner of direction-optimising BFS: go pull when the
// frontier's edges exceed the unvisited edges / alpha while the frontier is
// growing, leave pull when the frontier falls below n / beta.  (p.alpha is the
// tuned alpha scaled by 1 + 4 n / L2 bytes at launch.)
__device__ __forceinline__ int heuristic_variant(const LoopParams& p, int prev_variant, long long count,
                                                 long long prev_count, long long edges,
                                                 long long unvisited_edges, bool small_rows) {
  bool pull;
  if (prev_variant == BFS_VARIANT_PULL) pull = (float)count * p.beta >= (float)p.n;
  else pull = (float)edges * p.alpha > (float)unvisited_edges && count >= prev_count;
  if (pull) return BFS_VARIANT_PULL;
  // a small frontier of short rows: one warp per vertex beats the binning's scan
  return (count <= p.small_frontier && small_rows) ? BFS_VARIANT_TD_WARP : BFS_VARIANT_TD_BINNED;
}

constexpr size_t kFlatBytes = (sizeof(FlatSmem) + 15) / 16 * 16;
// the largest phase's area, without and with the tiled phase
constexpr size_t kPhaseBytes = std::max(sizeof(PullSmem), kFlatBytes);
static_assert(offsetof(Smem, cl) + offsetof(Claims, cq) + kLongQ * sizeof(int) <= sizeof(Smem) + kPhaseBytes,
              "the long claim buffer ends with the phases' area");
constexpr size_t kMlpBytes = (sizeof(float) * BFS_MLP_PARAMS + 15) / 16 * 16;
static_assert(kPhaseBytes >= kMlpBytes + sizeof(bfsdev::MlpScratch), "the network fits the phases' area");
constexpr size_t kTiledBytes = std::max(kPhaseBytes, kFlatBytes + sizeof(uint32_t) * 3 * kTileWordsMax);

// Brings the selector network's parameters to shared memory during a barrier.
template <bool kLearned>
struct FetchMlp {
  float* dst;
  const float* src;
  __device__ void start() const {
    if constexpr (kLearned) {
      static_assert(BFS_MLP_PARAMS % 4 == 0, "whole 16-byte groups");
      for (int i = threadIdx.x; i < BFS_MLP_PARAMS / 4; i += kBlock)
        asm volatile("cp.async.ca.shared.global [%0], [%1], 16;" ::"r"(smem_addr(dst + 4 * i)), "l"(src + 4 * i) : "memory");
    }
  }
  __device__ void finish() const {
    if constexpr (kLearned) asm volatile("cp.async.wait_all;" ::: "memory");
  }
};

// kTiles: the kernel can run the tiled phase.  Runs that cannot pick the tiled
// variant launch the instance without it: on R-MAT scale 26 the tiled phase's
// code alone made the other phases 5 % slower.
// kLearned: the selector network may choose the variants.  Learned runs never
// pick the tiled variant, and the other runs do without the network's code.
// kLong: see topdown_phase; for forced and scheduled runs, which may run a large level
// by threads or warps.  The heuristic runs only levels of at most 32 edges a warp that
// way, and the network's choices at large levels are others.  Six roots on 2^27 edges,
// every level by threads and by warps, ms per root: edgefactor 4 15.2 -> 11.1 and 13.1 ->
// 7.6, 8 7.9 -> 7.8 and 6.5 -> 6.0, 16 6.7 and 4.5 as before (with a buffer of 6,144 entries in
// every instance, which took L1 from every phase, edgefactor 4 took 14.0 and 11.9).
template <bool kTiles, bool kLearned, bool kLong>
__global__ void __launch_bounds__(kBlock, 2) level_loop_kernel(LoopParams p) {
  // dynamic shared memory: one area that the phases use in turn (PullSmem, or
  // FlatSmem and the tiled phase's 3 * kTileWordsMax words), and between phases
  // the selector network's parameters
  extern __shared__ __align__(64) unsigned char s_all[];
  // kLong: the CTA's state lies in front of the phases' area, so that its claim buffer can go on into it
  __shared__ std::conditional_t<kLong, char, Smem> s_state;
  Smem& sm = *reinterpret_cast<Smem*>(kLong ? s_all : reinterpret_cast<unsigned char*>(&s_state));
  unsigned char* const s_dyn = kLong ? s_all + sizeof(Smem) : s_all;
  FlatSmem& s_flat = *reinterpret_cast<FlatSmem*>(s_dyn);
  uint32_t* s_tile = reinterpret_cast<uint32_t*>(s_dyn + kFlatBytes);
  PullSmem& s_pull = *reinterpret_cast<PullSmem*>(s_dyn);
  [[maybe_unused]] float* const s_mlp = reinterpret_cast<float*>(s_dyn);
  [[maybe_unused]] bfsdev::MlpScratch& s_mlp_scratch = *reinterpret_cast<bfsdev::MlpScratch*>(s_dyn + kMlpBytes);
  const int tid = threadIdx.x;
  unsigned long long bar_target = 0;
  if (tid == 0) {
    bar_target = bfsdev::barrier_base(p.bar, gridDim.x);
    sm.owner = -1;
    claims_reset(sm.cl);
    sm.acc[0] = sm.acc[1] = sm.acc[2] = sm.acc[3] = 0;
  }
  // The network's parameters come to the phases' area during every barrier, when
  // it is free.  Kept in 21 KB of their own they left the expansion half the L1
  // (learned runs, in their own 21 KB against brought at each barrier: 4 roots at scale 26 5,880 us and 5,635, scale
  // 21 442 and 413, Erdos-Renyi 1 M 232 and 222; grid 128^3, all narrow levels, 2,702 and 2,763).
  const FetchMlp<kLearned> fetch_mlp{s_mlp, p.mlp};

  const long long gtid = (long long)blockIdx.x * kBlock + tid;
  const long long gthreads = (long long)gridDim.x * kBlock;
  const unsigned nblocks = gridDim.x;

  // ---- init: outputs to -1, bitmaps cleared, counters zeroed.  Vertices
  // without edges (and the tail beyond n) start as visited, since no traversal
  // can reach them.  A single source is seeded in the same phase; several
  // sources (ragged runs) get a seeding phase of their own.  The output fill
  // only stores and the bitmap loop's loads are independent, so neither waits
  // on a load per step.
  const bool single = p.nsources == 1;
  const int s0 = p.src0;
  // outputs: 4 vertices per thread and step, one 16-byte store each when aligned
  const bool vec = ((reinterpret_cast<uintptr_t>(p.level) | reinterpret_cast<uintptr_t>(p.parent)) & 15u) == 0;
  const long long n4 = ((long long)p.n + 3) / 4;
  for (long long q = gtid; q < n4; q += gthreads) {
    const long long v = 4 * q;
    int lv[4], pv[4];
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      const bool src = single && v + c == s0;
      lv[c] = src ? 0 : -1;
      pv[c] = src ? s0 : -1;
    }
    if (vec && v + 4 <= p.n) {
      *reinterpret_cast<int4*>(p.level + v) = make_int4(lv[0], lv[1], lv[2], lv[3]);
      *reinterpret_cast<int4*>(p.parent + v) = make_int4(pv[0], pv[1], pv[2], pv[3]);
    } else {
      for (int c = 0; c < 4 && v + c < p.n; ++c) {
        p.level[v + c] = lv[c];
        p.parent[v + c] = pv[c];
      }
    }
  }
  // bitmaps: vis starts as the edgeless vertices (and the tail beyond n) plus
  // the single source; one thread per word when the dead bits are precomputed
  const uint32_t srcbit = 1u << (s0 & 31);
  const long long sw = s0 >> 5;
  if (p.dead != nullptr) {
    for (long long w = gtid; w < p.nwords; w += gthreads) {
      const bool sword = single && w == sw;
      p.vis[w] = __ldg(&p.dead[w]) | (sword ? srcbit : 0u);
      p.bits[0][w] = sword ? srcbit : 0u;
      p.bits[1][w] = 0;
      p.bits[2][w] = 0;
    }
  } else {  // dead bits from the row offsets, one warp per word
    const long long nv32 = (long long)p.nwords * 32;
    for (long long v = gtid; v < nv32; v += gthreads) {
      const bool dead = v >= p.n || (single && v == s0) || __ldg(&p.toff[v + 1]) == __ldg(&p.toff[v]);
      const unsigned dm = __ballot_sync(kFull, dead);
      if ((tid & 31) == 0) {
        const long long w = v >> 5;
        const bool sword = single && w == sw;
        p.vis[w] = dm;
        p.bits[0][w] = sword ? srcbit : 0u;
        p.bits[1][w] = 0;
        p.bits[2][w] = 0;
      }
    }
  }
  if (blockIdx.x == 0) {
    static_assert(kCtrRing * sizeof(LevelCtr) / 8 <= kBlock, "one word of the ring per thread");
    if (tid < kCtrRing * (int)(sizeof(LevelCtr) / 8)) reinterpret_cast<unsigned long long*>(p.ctr)[tid] = 0ull;
    __syncthreads();
    if (single && tid == 0) {
      p.queue[0][0] = s0;
      const long long deg = __ldg(&p.off[s0 + 1]) - __ldg(&p.off[s0]);
      p.ctr[0].count = 1;
      p.ctr[0].edges = (unsigned long long)deg;
      p.ctr[0].bins[deg <= 32 ? 0 : (deg <= 1024 ? 1 : 2)] = 1;
      if (deg > p.chunk_deg) push_chunks(p, 0, s0, deg);
    }
  }
  if (!bfsdev::grid_barrier(p.bar, nblocks, bar_target, p.spin_limit, p.status, FetchCtr{&p.ctr[0], &sm.ctr}, fetch_mlp))
    return;

  if (!single) {  // seed level 0 with the sources (block 0)
    if (blockIdx.x == 0) {
      Acc acc;
      for (int i = tid; i < p.nsources; i += kBlock) {
        const int s = p.sources[i];
        p.level[s] = 0;
        p.parent[s] = s;
        atomicOr(&p.bits[0][s >> 5], 1u << (s & 31));
        p.queue[0][i] = s;
        const long long deg = __ldg(&p.off[s + 1]) - __ldg(&p.off[s]);
        acc_vertex(acc, deg);
        if (deg > p.chunk_deg) push_chunks(p, 0, s, deg);
      }
      if (tid == 0) p.ctr[0].count = (unsigned)p.nsources;
      end_phase(p, 0, acc, sm);
    }
    if (!bfsdev::grid_barrier(p.bar, nblocks, bar_target, p.spin_limit, p.status, FetchCtr{&p.ctr[0], &sm.ctr}, fetch_mlp))
      return;
  }

  // ---- level loop
  long long cum_count = 0, cum_edges = 0;
  int prev_variant = -1;
  unsigned prev_count = 0;
  int clr_first = -1;
  uint64_t t_prev = 0;
  if (blockIdx.x == 0 && tid == 0) t_prev = bfsdev::global_timer_ns();
  int k = 0;
  Acc acc;
  for (;; ++k) {
    PHASE_TS(k, 0);
    const LevelCtr& c = sm.ctr;  // (the next fetch comes after this level's work and a CTA barrier)
    const unsigned count = c.count;
    const unsigned nchunks = c.chunks;
    const long long edges = (long long)c.edges;
    const bool big_rows = (c.bins[1] | c.bins[2]) != 0;
    const bool sparse_clr = k >= 1 && (long long)prev_count * 4 < p.nwords;
    const int32_t* PQ = p.queue[(k + 2) % 3];
    if (count == 0) break;
    cum_count += count;
    cum_edges += edges;
    const long long unvisited = (long long)p.n - cum_count;
    const long long unvisited_edges = p.nnz - cum_edges;

    // A level whose frontier has few edges runs on the first half of the CTAs
    // (one per SM when two are resident): only they recycle, expand and arrive
    // at its barrier, which halves the barrier's arrivals and the CTAs that
    // contend for the level's few claims.  The other CTAs still choose the
    // variant (the next level's choice depends on it) and wait at the barrier.
    // A CTA that does not arrive may fall behind the others, which must not clear the
    // counters that it has yet to read: every kAllArrive-th level is everyone's.
    constexpr int kAllArrive = 32, kClearAhead = 4;
    static_assert(kAllArrive + kClearAhead < kCtrRing, "no slot is cleared before the last CTA has read it");
    const bool narrow = edges <= p.narrow_edges && nblocks >= 2 && k % kAllArrive != kAllArrive - 1;
    const unsigned G = narrow ? (nblocks + 1) / 2 : nblocks;
    const bool part = blockIdx.x < G;
    const long long pthreads = (long long)G * kBlock;

    // recycle: counters of level k+4, bitmap of level k-1 (stores only; they
    // drain while the selector runs)
    if (blockIdx.x == 0 && tid < (int)(sizeof(LevelCtr) / 8))
      reinterpret_cast<unsigned long long*>(&p.ctr[(k + kClearAhead) % kCtrRing])[tid] = 0ull;
    if (k >= 1 && part) {
      uint32_t* clr = p.bits[(k + 2) % 3];
      if (sparse_clr) {
        if (clr_first >= 0) clr[clr_first >> 5] = 0u;
        for (long long i = gtid + pthreads; i < prev_count; i += pthreads) clr[PQ[i] >> 5] = 0u;
      } else {
        for (long long w = gtid; w < p.nwords; w += pthreads) clr[w] = 0u;
      }
    }
    PHASE_TS(k, 1);

    int variant;
    FirstRow first;
    if constexpr (kLearned) {
      // every CTA evaluates the network (all compute the same bits)
      // The last four warps compute the outputs, about 0.9 us of latencies; meanwhile each other warp fetches the
      // row it starts with if the level goes a warp per vertex (a narrow level's vertices all sit in those warps).
      if (tid >= kBlock - bfsdev::kMlpThreads) {
        learned_outputs(p, s_mlp, s_mlp_scratch, &sm.mlp_y.x, tid - (kBlock - bfsdev::kMlpThreads), k, c, unvisited,
                        unvisited_edges);
      } else if (part && blockIdx.x + (unsigned)(tid >> 5) * G < count) {
        first.u = p.queue[k % 3][blockIdx.x + (unsigned)(tid >> 5) * G];
        first.b = __ldg(&p.off[first.u]);
        first.e = __ldg(&p.off[first.u + 1]);
      }
      __syncthreads();  // the outputs are there, and the network's area is free for the phase
      variant = bfsdev::mlp_argmin(sm.mlp_y);
    } else if (p.selector == BFS_SELECT_FORCED) {
      variant = p.forced;
    } else if (p.selector == BFS_SELECT_SCHEDULE && k < p.schedule_len) {
      variant = p.schedule[k];
    } else {
      variant = heuristic_variant(p, prev_variant, count, prev_count, edges, unvisited_edges, !big_rows);
    }
    if (variant < 0 || variant >= BFS_NUM_VARIANTS) variant = BFS_VARIANT_TD_BINNED;
    if (variant == BFS_VARIANT_TILED && (!kTiles || p.t_jc == nullptr)) variant = BFS_VARIANT_PULL;  // the SpMV untiled
    PHASE_TS(k, 2);
    if (part) {
      if (variant == BFS_VARIANT_PULL) pull_phase(p, k, count, sm, s_pull, acc, G);
      else if (kTiles && variant == BFS_VARIANT_TILED) tiled_phase(p, k, sm, s_flat, s_tile, acc, G);
      // the degree-binned variant deals a small frontier's edges out flat
      else if (variant == BFS_VARIANT_TD_BINNED && count <= (unsigned)kFlatRows && edges <= p.flat_visits * pthreads)
        flat_phase(p, k, count, sm, s_flat, acc, G);
      else topdown_phase<kLong>(p, k, variant, count, nchunks, first, sm, s_flat, acc, G);
      PHASE_TS(k, 3);
      end_phase(p, k + 1, acc, sm, claim_room<kLong>(variant));
    }
    PHASE_TS(k, 4);
    PHASE_ARRIVAL(k);
    // the first entry of f_k that this thread clears in the next level: in flight across the barrier
    clr_first = gtid < count ? p.queue[k % 3][gtid] : -1;
    const int4 level_bins = p.want_stats && blockIdx.x == 0 && tid == 0
                                ? make_int4((int)c.bins[0], (int)c.bins[1], (int)c.bins[2], 0)
                                : make_int4(0, 0, 0, 0);
    if (!bfsdev::grid_barrier_partial(p.bar, G, bar_target, p.spin_limit, p.status,
                                      FetchCtr{&p.ctr[(k + 1) % kCtrRing], &sm.ctr}, fetch_mlp))
      return;
    PHASE_TS(k, 6);

    if (p.want_stats && blockIdx.x == 0 && tid == 0 && k < kMaxStatLevels) {
      const uint64_t t = bfsdev::global_timer_ns();
      bfs_level_stat st;
      st.frontier_count = count;
      st.frontier_edges = edges;
      st.bin_count[0] = level_bins.x;
      st.bin_count[1] = level_bins.y;
      st.bin_count[2] = level_bins.z;
      st.unvisited_count = unvisited;
      st.unvisited_edges = unvisited_edges;
      st.time_ns = (int64_t)(t - t_prev);
      st.variant = variant;
      st.reserved = 0;
      p.stats[k] = st;
      t_prev = t;
    }
    prev_variant = variant;
    prev_count = count;
  }

  if (gtid == 0) {
    bfsdev::barrier_pad(p.bar, nblocks, bar_target);  // partial barriers: round the counter to the grid size
    p.misc[0] = k;
    *p.edges_out = p.directed ? cum_edges : cum_edges / 2;  // arcs, or undirected edges
  }
  // ragged: copy the union-space outputs into each part's arrays, local ids.  One pass over the union with four
  // vertices of a thread in flight: bound by loads that hit L2 and by the stores.  A pass per part kept the grid
  // waiting for each part's loads in turn (32 parts of 2^12 to 2^20 vertices, whole call: 417 -> 383 us).
  if (p.part_out != nullptr) {
    constexpr int kFlight = 4;
    for (long long v0 = gtid; v0 < p.n; v0 += kFlight * gthreads) {
      int lev[kFlight], par[kFlight];
#pragma unroll
      for (int j = 0; j < kFlight; ++j) {
        const long long v = v0 + j * gthreads;
        if (v < p.n) {
          lev[j] = p.level[v];
          par[j] = p.parent[v];
        }
      }
      int q = 0;
#pragma unroll
      for (int j = 0; j < kFlight; ++j) {
        const long long v = v0 + j * gthreads;
        if (v >= p.n) break;
        int last = p.parts - 1;  // v's part: the last one that starts at or before v (v grows with j, so q only rises)
        while (q < last) {
          const int mid = (q + last + 1) / 2;
          if (p.part_base[mid] <= v) q = mid;
          else last = mid - 1;
        }
        const long long base = p.part_base[q];
        p.part_out[q][v - base] = lev[j];
        p.part_out[p.parts + q][v - base] = par[j] >= 0 ? (int)(par[j] - base) : -1;
      }
    }
  }
}

}  // namespace

#ifdef BFS_PHASE_TIMING
extern "C" __attribute__((visibility("default"))) int bfs_debug_phase_times(unsigned long long* host, int levels) {
  if (levels > 4096) levels = 4096;
  cudaDeviceSynchronize();
  if (cudaMemcpyFromSymbol(host, g_phase_ts, sizeof(unsigned long long) * 8 * levels) != cudaSuccess) return 1;
  static unsigned long long zero[4096][8];
  cudaMemcpyToSymbol(g_phase_ts, zero, sizeof(zero));
  return 0;
}
#endif

int launch_level_loop(const RunRequest& r, cudaStream_t s) {
  bfs_graph* g = r.g;
  Workspace* w = r.w;
  DeviceInfo di;
  if (int e = current_device_info(&di)) return e;
  if (r.nsources < 1 || r.nsources > kMaxSources) return fail(BFS_ERR_INVALID_ARG, "number of sources out of range");
  int sched_len = 0;
  const bool need_sched = r.selector == BFS_SELECT_SCHEDULE && r.h_schedule && r.schedule_len > 0;
  if (r.nsources > 1 || need_sched) {  // stage through pinned memory (no pageable-copy synchronisation)
    if (int e = stage_wait(w)) return e;
    if (r.nsources > 1) {
      std::copy(r.h_sources, r.h_sources + r.nsources, w->h_stage + kMaxSchedule);
      BFS_CUDA_TRY(cudaMemcpyAsync(w->sources, w->h_stage + kMaxSchedule, sizeof(int32_t) * r.nsources,
                                   cudaMemcpyHostToDevice, s));
    }
    if (need_sched) {
      sched_len = r.schedule_len < kMaxSchedule ? r.schedule_len : kMaxSchedule;
      std::copy(r.h_schedule, r.h_schedule + sched_len, w->h_stage);
      BFS_CUDA_TRY(cudaMemcpyAsync(w->schedule, w->h_stage, sizeof(int32_t) * sched_len, cudaMemcpyHostToDevice, s));
    }
    BFS_CUDA_TRY(cudaEventRecord(w->stage_ev, s));
  }
  if (!g->d_off || !g->d_toff || (g->nnz > 0 && (!g->d_adj || !g->d_tadj)))
    return fail(BFS_ERR_INVALID_ARG, "graph without rows");
  const bfs_tuning t = effective_tuning(g);
  // the tiled variant needs the graph's tiles: built here the first time a run may use it
  bool may_tile = r.selector == BFS_SELECT_FORCED && r.forced == BFS_VARIANT_TILED;
  for (int i = 0; i < sched_len && !may_tile; ++i) may_tile = r.h_schedule[i] == BFS_VARIANT_TILED;
  const TileSet* tiles = r.tiles;
  if (may_tile && tiles == nullptr) {
    TileSet* ts = nullptr;
    if (int e = ensure_tiles(g, s, &ts)) return e;
    tiles = ts;
  }
  LoopParams p{};
  p.off = g->d_off;
  p.adj = g->d_adj;
  p.toff = g->d_toff;
  p.tadj = g->d_tadj;
  p.directed = g->directed ? 1 : 0;
  p.dead = g->d_dead;
  p.n = g->n;
  p.nwords = w->nwords;
  p.nnz = g->nnz;
  p.level = r.level;
  p.parent = r.parent;
  for (int i = 0; i < 3; ++i) {
    p.queue[i] = w->queue[i];
    p.bits[i] = w->bits[i];
  }
  p.vis = w->vis;
  p.chunks[0] = w->chunks[0];
  p.chunks[1] = w->chunks[1];
  p.chunk_cap = w->chunk_cap;
  p.ctr = w->ctr;
  p.status = w->status;
  p.stats = w->stats;
  p.misc = w->misc;
  p.edges_out = w->edges_out;
  p.sources = w->sources;
  p.src0 = r.h_sources[0];
  p.nsources = r.nsources;
  p.selector = r.selector;
  p.forced = r.forced;
  p.schedule = w->schedule;
  p.schedule_len = sched_len;
  p.mlp = r.selector == BFS_SELECT_LEARNED ? learned_params_device(s) : nullptr;
  graph_feature_constants(g->n, g->nnz, &p.feat_log_n, &p.feat_log_nnz, &p.feat_inv_n, &p.feat_inv_nnz);
  p.want_stats = r.want_stats ? 1 : 0;
  p.spin_limit = r.spin_limit ? r.spin_limit : (1u << 25);
  p.warp_deg = t.warp_degree;
  p.cta_deg = t.cta_degree;
  p.pull_thread_deg = t.pull_thread_degree;
  p.chunk_deg = t.chunk_degree;
  // top-down's atomics on the parent array get dearer once 4 bytes per vertex
  // no longer fit in L2, so the switch to pull comes earlier on large graphs
  p.alpha = (float)(t.alpha * (1.0 + 4.0 * (double)g->n / (double)(di.l2_bytes > 0 ? di.l2_bytes : (1ll << 27))));
  p.beta = t.beta;
  p.parts = g->parts;
  p.part_base = g->d_part_base;
  p.part_out = r.part_out;
  if (may_tile && tiles != nullptr) {
    const TileSet* ts = tiles;
    p.t_jc = ts->jc;
    p.t_cp = ts->cp;
    p.t_ir = ts->ir;
    p.t_dir_jc = ts->tdir_jc;
    p.t_dir_ir = ts->tdir_ir;
    p.t_rb_bits = ts->rb_bits;
    p.t_cb_bits = ts->cb_bits;
    p.t_nrb = ts->nrb;
    p.t_ncb = ts->ncb;
  }

  // The long claim buffer (kLong) pays where a level can overfill the short ones of all CTAs together: below twice
  // their entries (2.6 M vertices) it gained nothing (2.1 M, edgefactor 64: 5.4 and 2.7 ms with either) and cost
  // narrow levels 0.5 % (grid 128^3, all by warps: 2.660 and 2.675 ms).
  const bool picked = r.selector == BFS_SELECT_FORCED || r.selector == BFS_SELECT_SCHEDULE;
  const bool long_buffer = p.t_jc || (picked && g->n > 2ll * (2 * di.sm_count) * kQBuf);
  const size_t dyn_smem = (p.t_jc ? kTiledBytes : kPhaseBytes) + (long_buffer ? sizeof(Smem) : 0);
  const void* const kernels[] = {
      (const void*)level_loop_kernel<false, false, false>, (const void*)level_loop_kernel<false, false, true>,
      (const void*)level_loop_kernel<true, false, true>, (const void*)level_loop_kernel<false, true, false>};
  const void* kernel = kernels[p.mlp ? 3 : p.t_jc ? 2 : long_buffer ? 1 : 0];
  {  // the attribute belongs to the current device: set it once per device
    static std::mutex mu;
    static bool configured[64] = {};
    std::lock_guard<std::mutex> lk(mu);
    if (di.device < 0 || di.device >= 64) return fail(BFS_ERR_UNSUPPORTED, "device ordinal out of range");
    if (!configured[di.device]) {
      for (const void* f : kernels)
        BFS_CUDA_TRY(cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                          (int)(sizeof(Smem) + kTiledBytes)));
      configured[di.device] = true;
    }
  }
  int per_sm = 0;
  BFS_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, kBlock, dyn_smem));
  if (per_sm < 1) return fail(BFS_ERR_CUDA, "level loop kernel cannot be resident");
  const int grid = (t.ctas_per_sm > 0 ? std::min(per_sm, t.ctas_per_sm) : per_sm) * di.sm_count;
  if (int e = prepare_barrier(w, 0, grid, s, &p.bar)) return e;
  p.small_frontier = t.small_frontier > 0 ? t.small_frontier : (t.small_frontier == 0 ? (long long)grid * kWarps : 0);
  p.probe = g->d_probe;
  p.rank = g->d_rank;
  // A claim by the parent's old value saves the bitmap look-up and one of two atomics with a result, on words
  // that conflict less (Erdos-Renyi, n = 1 M, 77 K-vertex level: 32 -> 27 us; grid 128^3: 2.56 -> 2.50 ms); once
  // the parents no longer sit in L2 its result comes from DRAM (scale 26, 7 M edges: 425 -> 496 us).
  p.claim_by_parent = 4ll * g->n <= (di.l2_bytes > 0 ? di.l2_bytes : (1ll << 27)) / 2;
  // 32 parts of a ragged batch, 0.9 M edges: flat 28 us, by rows and chunks 55 us; at scale 26, 2.1 M edges, the
  // chunks' two visits in flight win (171 us against 223).  Whole traversals feel it by 1 or 2 % at most: 16 against 4,
  // us per root over 32 roots, edgefactor 16, scale 20 72.1 and 73.0, 22 127.2 and 127.6, 24 419.5 and 420.8, 25 794
  // and 794, 26 1,489.5 and 1,488.5; 32 ragged parts 417 and 436; against it scale 24 with edgefactor 64, 513 and 509
  p.flat_visits = p.claim_by_parent ? 16 : 4;
  // one chunk per resident warp while a lane per word allows it (see pull_phase)
  const long long grid_warps = (long long)grid * kWarps;
  p.pull_words = (int)std::min<long long>(32, std::max<long long>(1, (w->nwords + grid_warps - 1) / grid_warps));
  while (((long long)g->n - 1) >> p.fr_shift >= 32ll * kFrWords) ++p.fr_shift;
  // every CTA reads the whole queue to build the summary: at most 8,192 vertices (12 % of its bits set; a
  // limit of 32,768 measured the same), and few against n so that the rows' scans pay for it
  p.fr_limit = (unsigned)std::min<long long>(8192, g->n / 128);
  p.narrow_edges = t.narrow_edges > 0 ? t.narrow_edges : (t.narrow_edges == 0 ? (1ll << 14) : -1);
#ifdef BFS_PHASE_TIMING
  fprintf(stderr, "level loop: %d CTAs (%d per SM), %zu bytes dynamic shared memory\n", grid, per_sm, dyn_smem);
#endif
  void* args[] = {&p};
  BFS_CUDA_TRY(cudaLaunchCooperativeKernel(kernel, dim3(grid), dim3(kBlock), args, dyn_smem, s));
  return BFS_OK;
}

}  // namespace bfsint
