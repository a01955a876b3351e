// Batched BFS: up to 64 roots in one persistent traversal.
//
// Every vertex carries 64-bit words: F_k[v] (bit r set when v is in the
// frontier of root r at level k), V[v] (bit r set when root r has reached v)
// and F_{k+1}[v].  One level is the boolean sparse matrix-dense matrix product
// F_{k+1} = (A (x) F_k) AND NOT V, i.e. the SpMSV of Sec. 3.2 for 64 vectors at
// once.  Parents follow the same max-id rule as the single-root traversal: for
// a vertex v newly reached by root r, parent_r[v] is the largest neighbour u
// with bit r in F_k[u], found by scanning v's sorted row from the largest id
// down and masking off the bits already resolved.
//
// "Reached before level k+1" is tested as V | F_k, so V only has to absorb a
// frontier's bits during the level that expands it, and every level is one
// phase.  Two ways to expand a level (identical results):
//   pull     : every vertex not yet reached by all roots scans its row, first
//              the top eight entries of eight rows at a time, then row by row
//              with the whole warp; lane r owns root r (and r + 32) and takes
//              its parent from a bit transpose of the entries' words; rows above
//              kChunkEdges entries go in kChunkEdges-entry chunks (a static table
//              built with the graph), one warp per chunk, the chunks combining
//              through atomicMax on the parents and atomicOr on F_{k+1};
//   top-down : every frontier row ORs its bits into F_{k+1} of unreached
//              neighbours and offers itself as their parent with atomicMax
//              for each new root bit (every frontier neighbour offers, so the
//              largest id wins); the first writer of any bit enqueues the
//              neighbour.
//              Rows above kChunkEdges entries are split into chunk items.
// Output rows are root-major: level[r * n + v], parent[r * n + v].  During
// the traversal the parents go to vertex-major scratch (sp[v][r], one row of
// `stride` ints per vertex), so that the results of one vertex share a few
// sectors instead of landing 4 * n bytes apart, and the levels to bit planes:
// bit r of plane[j][v] is bit j of root r's level of v, so that a level costs
// a vertex one word per set bit of its number and an R-MAT traversal three
// words per vertex in all, where 64 ints would be 256 bytes.  The planes take
// F_k's level when level k expands it (by the vertex's owner, without atomics).
// A last phase turns both into the outputs, coalesced.
//
// The words are 8, 16, 32 or 64 bits wide (one bit per root of the
// traversal; bit arithmetic is done in 64-bit registers whatever the word).
// 64 is the default: a traversal's row scans cost about the same whatever
// the number of roots it carries, so fewer, wider traversals win even when
// the frontier array no longer fits in L2 (measured at scales 22 to 26).
#include <cooperative_groups.h>
#include <climits>

#include "claims.cuh"
#include "device_common.cuh"
#include "internal.h"

namespace cg = cooperative_groups;

namespace bfsint {
namespace {

using bfsdev::kFull;

// What bounds the kernel and why it is split this way (R-MAT scale 24, 64
// roots, level times): the pull levels look up one frontier word per row entry
// in an array that just exceeds L2, with 32 warps per SM to hide the latency
// (halving them makes the levels 1.4 times slower), and spend as many
// instructions on recording parents as on finding them.  Recording was the
// larger part when a lane or a warp wrote one root's level and parent at a
// time (4-byte stores 256 bytes apart): with a lane per root the two dense
// levels went from 9.4 and 5.9 ms to 4.0 and 2.9 ms.  The loads in flight
// below are the best of 1 to 4 each; deeper ones cost registers that spill.
constexpr int kBBlock = 512;
static_assert(kBBlock == kClaimBlock, "the claim buffers assume 512-thread CTAs");
constexpr int kBWarps = kBBlock / 32;
constexpr int kTop = 8;        // entries of a row examined in the first packed step, 32 / kTop rows per load
constexpr int kNext = 32;      // entries of a row examined in the second, one row per load
constexpr int kTopLoads = 2, kNextLoads = 2;  // loads per lane in flight in these steps
constexpr int kRowLoads = 4;   // loads per lane in flight when the warp scans the rest of one row
constexpr int kFewBits = 6;    // up to this many new roots are resolved one by one instead of by a transpose
constexpr int kPlanes = 31;    // level bit planes: levels are below 2^31
static_assert(8 * kPlanes <= 64 * sizeof(int32_t), "the planes fit the second half of the scratch");

struct BatchParams {
  const int64_t* __restrict__ off;   // out-rows: top-down
  const int32_t* __restrict__ adj;
  const int64_t* __restrict__ toff;  // in-rows: pull (the same arrays when undirected)
  const int32_t* __restrict__ tadj;
  int32_t directed;
  int32_t n;
  long long nnz;
  int32_t k;  // roots in this traversal (<= 64)
  uint64_t mask;
  int32_t src[64];
  int32_t* level;   // [k][n]
  int32_t* parent;  // [k][n]
  void* planes;     // level bit planes, Word[kPlanes][n]
  int32_t* sp;      // scratch parents [n][stride]
  int32_t stride;   // roots per scratch row (the word width)
  const uint32_t* __restrict__ dead;  // bitmap of the vertices no arc enters
  void* F[3];  // Word[n] each
  void* V;     // Word[n]
  int32_t* queue[3];
  int64_t* chunks[2];
  long long chunk_cap;  // entries of each chunk list
  const int64_t* big;  // chunks of in-rows longer than kChunkEdges (static, per graph)
  long long nbig;
  LevelCtr* ctr;
  bfsdev::GridBarrier* bar;
  int* status;
  int32_t* misc;
  bfs_level_stat* stats;  // per-level statistics when non-null
  unsigned spin_limit;
  long long td_limit;
};

using Bits = unsigned long long;

// atomicOr of v into a word of an 8-, 16-, 32- or 64-bit array; returns the old word.
template <typename Word>
__device__ __forceinline__ Bits atomic_or_word(Word* a, Bits v) {
  if constexpr (sizeof(Word) == 8) {
    return atomicOr(reinterpret_cast<unsigned long long*>(a), v);
  } else if constexpr (sizeof(Word) == 4) {
    return atomicOr(reinterpret_cast<unsigned*>(a), (unsigned)v);
  } else {  // the aligned 32-bit word that holds *a
    const uintptr_t ad = reinterpret_cast<uintptr_t>(a);
    const int sh = (int)(ad & 3u) * 8;
    const unsigned old = atomicOr(reinterpret_cast<unsigned*>(ad & ~(uintptr_t)3), (unsigned)v << sh);
    return (Bits)((old >> sh) & ((1u << (8 * sizeof(Word))) - 1u));
  }
}

// OR of v over the warp (v has at most 8 * sizeof(Word) bits).
template <typename Word>
__device__ __forceinline__ Bits warp_or(Bits v) {
  const unsigned lo = __reduce_or_sync(kFull, (unsigned)v);
  if constexpr (sizeof(Word) == 8) {
    const unsigned hi = __reduce_or_sync(kFull, (unsigned)(v >> 32));
    return ((Bits)hi << 32) | lo;
  } else {
    return lo;
  }
}

// 32 x 32 bit transpose over the warp: bit s of lane r's result is bit r of lane s's x.
__device__ __forceinline__ unsigned transpose32(unsigned x, int lane) {
#pragma unroll
  for (int s = 16; s >= 1; s >>= 1) {
    const unsigned lo = s == 16 ? 0x0000ffffu : s == 8 ? 0x00ff00ffu : s == 4 ? 0x0f0f0f0fu : s == 2 ? 0x33333333u : 0x55555555u;
    const unsigned y = __shfl_xor_sync(kFull, x, s);
    x = (lane & s) ? ((x & ~lo) | ((y & ~lo) >> s)) : ((x & lo) | ((y & lo) << s));
  }
  return x;
}

// Records the parents of the roots found in one row: m0 (m1) has a bit for
// every slot of the row whose word holds root `lane` (`lane` + 32), the lowest
// slot being the largest id, and lane s holds slot s's id u.  kOffer: the ids
// are candidates of one chunk of the row, so they are offered with atomicMax.
// Returns the roots found (the same in every lane).
template <typename Word, bool kOffer>
__device__ __forceinline__ Bits store_parents(const BatchParams& p, int v, unsigned m0, unsigned m1, int u, int lane) {
  int32_t* row = p.sp + (long long)v * p.stride;
  const int u0 = __shfl_sync(kFull, u, m0 ? __ffs(m0) - 1 : 0);
  if (m0) {
    if (kOffer) bfsdev::red_max_i32(row + lane, u0);
    else row[lane] = u0;
  }
  Bits found = __ballot_sync(kFull, m0 != 0);
  if constexpr (sizeof(Word) == 8) {
    const int u1 = __shfl_sync(kFull, u, m1 ? __ffs(m1) - 1 : 0);
    if (m1) {
      if (kOffer) bfsdev::red_max_i32(row + lane + 32, u1);
      else row[lane + 32] = u1;
    }
    found |= (Bits)__ballot_sync(kFull, m1 != 0) << 32;
  }
  return found;
}

// The whole warp scans entries [b, t) of v's row from the top, 32 * kRowLoads
// per step, and resolves the roots in `need`; returns the bits found (the same
// value in every lane).  kOffer: see store_parents.
template <typename Word, bool kOffer>
__device__ __forceinline__ Bits resolve_row(const BatchParams& p, const Word* F, int v, long long b, long long t,
                                            Bits need, int lane) {
  Bits found = 0;
  for (; t > b && need; t -= 32 * kRowLoads) {
    int u[kRowLoads];
    Bits f[kRowLoads];
#pragma unroll
    for (int q = 0; q < kRowLoads; ++q) {
      const long long j = t - 1 - lane - 32 * q;
      u[q] = j >= b ? __ldg(&p.tadj[j]) : 0;
    }
#pragma unroll
    for (int q = 0; q < kRowLoads; ++q)
      f[q] = (t - 1 - lane - 32 * q >= b && bfsdev::in_range(p.status, bfsdev::kSiteBatchPull, u[q], p.n)) ? (Bits)__ldcg(&F[u[q]])
                                                                                                         : 0ull;
#pragma unroll
    for (int q = 0; q < kRowLoads; ++q) {
      const Bits mine = f[q] & need;
      Bits nb = warp_or<Word>(mine);
      if (!nb) continue;
      found |= nb;
      need &= ~nb;
      if (__popcll(nb) <= kFewBits) {
        for (; nb; nb &= nb - 1) {  // each new root takes the lowest lane holding its bit (the largest id)
          const int r = __ffsll((long long)nb) - 1;
          const unsigned who = __ballot_sync(kFull, (mine >> r) & 1ull);
          if (lane == __ffs(who) - 1) {
            int32_t* o = p.sp + (long long)v * p.stride + r;
            if (kOffer) bfsdev::red_max_i32(o, u[q]);
            else *o = u[q];
          }
        }
      } else {
        const unsigned m0 = transpose32((unsigned)mine, lane);
        const unsigned m1 = sizeof(Word) == 8 ? transpose32((unsigned)(mine >> 32), lane) : 0u;
        store_parents<Word, kOffer>(p, v, m0, m1, u[q], lane);
      }
    }
  }
  return found;
}

// Examines kSlots entries of every row with roots to find, below its first
// `skip`, 32 / kSlots rows per load and kLoads loads in flight: lane l's row
// has deg entries ending at e and `need` roots to find.  Adds the roots found
// to `found` and takes them from `need`.  list: 32 ints of the warp.
template <typename Word, int kSlots, int kLoads>
__device__ __forceinline__ void resolve_packed(const BatchParams& p, const Word* F, int v, int skip, int deg,
                                               long long e, Bits& need, Bits& found, int lane, int* list) {
  constexpr int kRows = 32 / kSlots;  // rows per load
  const bool open = need != 0 && deg > skip;
  const unsigned pm = __ballot_sync(kFull, open);
  if (!pm) return;
  const int rows = __popc(pm);
  if (open) list[__popc(pm & bfsdev::lanemask_lt())] = lane;
  __syncwarp();
  Bits got = 0;
  const int sub = lane / kSlots, slot = skip + lane % kSlots;
  for (int base = 0; base < rows; base += kRows * kLoads) {
    int u[kLoads], own[kLoads];
    Bits f[kLoads];
    bool has[kLoads];
#pragma unroll
    for (int q = 0; q < kLoads; ++q) {
      const int i = base + q * kRows + sub;
      own[q] = list[min(i, rows - 1)];
      const int d = __shfl_sync(kFull, deg, own[q]);
      const long long eo = __shfl_sync(kFull, e, own[q]);
      has[q] = i < rows && slot < d;
      u[q] = has[q] ? __ldg(&p.tadj[eo - 1 - slot]) : 0;
    }
#pragma unroll
    for (int q = 0; q < kLoads; ++q)
      f[q] = (has[q] && bfsdev::in_range(p.status, bfsdev::kSiteBatchPull, u[q], p.n)) ? (Bits)__ldcg(&F[u[q]]) : 0ull;
#pragma unroll
    for (int q = 0; q < kLoads; ++q) {
      const Bits mine = f[q] & __shfl_sync(kFull, need, own[q]);
      const unsigned any = __ballot_sync(kFull, mine != 0);
      if (!any) continue;
      const unsigned m0 = transpose32((unsigned)mine, lane);
      const unsigned m1 = sizeof(Word) == 8 ? transpose32((unsigned)(mine >> 32), lane) : 0u;
#pragma unroll
      for (int j = 0; j < kRows; ++j) {
        const unsigned seg = (kSlots == 32 ? kFull : (1u << kSlots) - 1u) << (j * kSlots);
        if (!(any & seg)) continue;
        const int o = __shfl_sync(kFull, own[q], j * kSlots);
        const Bits fr =
            store_parents<Word, false>(p, __shfl_sync(kFull, v, o), m0 & seg, m1 & seg, u[q], lane);
        if (lane == o) got = fr;
      }
    }
  }
  need &= ~got;
  found |= got;
  __syncwarp();  // the list is free again
}

// Resolves 32 vertices against frontier F: lane l's vertex v has a row of deg
// entries ending at e and `need` roots to find.  First the top kTop entries of
// every row, 32 / kTop rows per load: a dense level ends most rows there, and
// short rows fill the lanes that a row each would leave idle; then the next
// kNext entries, a row per load; then row by row.  Returns the lane's bits found.
template <typename Word>
__device__ __forceinline__ Bits resolve_group(const BatchParams& p, const Word* F, int v, int deg, long long e,
                                              Bits need, int lane, int* list) {
  Bits found = 0;
  resolve_packed<Word, kTop, kTopLoads>(p, F, v, 0, deg, e, need, found, lane, list);
  resolve_packed<Word, kNext, kNextLoads>(p, F, v, kTop, deg, e, need, found, lane, list);
  for (unsigned lm = __ballot_sync(kFull, need != 0 && deg > kTop + kNext); lm; lm &= lm - 1u) {
    const int l = __ffs(lm) - 1;
    const long long el = __shfl_sync(kFull, e, l);
    const Bits fr = resolve_row<Word, false>(p, F, __shfl_sync(kFull, v, l), el - __shfl_sync(kFull, deg, l),
                                             el - kTop - kNext, __shfl_sync(kFull, need, l), lane);
    if (lane == l) found |= fr;
  }
  return found;
}

// Adds level k of the roots in F_k[v] = bits to the bit planes; called once per
// level and vertex, by the vertex's owner in that level.
template <typename Word>
__device__ __forceinline__ void add_level(const BatchParams& p, int v, Bits bits, int k) {
  for (unsigned m = (unsigned)k; m; m &= m - 1u) {
    Word* a = static_cast<Word*>(p.planes) + (long long)(__ffs(m) - 1) * p.n + v;
    *a = (Word)((Bits)*a | bits);
  }
}

// Top-down visit of edge (u -> w) with frontier bits f of u at level knext - 1.
template <typename Word>
__device__ __forceinline__ void td_visit(const BatchParams& p, const Word* Fc, Word* Fn, const Word* V, int knext,
                                         uint64_t f, int u, int w, Claims& cl) {
  if (!bfsdev::in_range(p.status, bfsdev::kSiteBatchTopDown, w, p.n)) return;
  const uint64_t nb = f & ~((Bits)V[w] | (Bits)Fc[w]);
  if (!nb) return;
  // u is a parent candidate of w for every new root bit (the offers return
  // nothing, so none of them is waited for)
  for (uint64_t b = nb; b; b &= b - 1) bfsdev::red_max_i32(&p.sp[(long long)w * p.stride + __ffsll((long long)b) - 1], u);
  if (((Bits)Fn[w] & nb) == nb) return;
  const Bits old = atomic_or_word(&Fn[w], nb);
  if (old == 0) {
    cta_enqueue(p, knext, cl, w);
    const long long deg = __ldg(&p.off[w + 1]) - __ldg(&p.off[w]);
    if (deg > kChunkEdges) push_chunks_cta(p, knext, cl, w, deg);
  }
}

// Pull over one kChunkEdges-entry chunk [rb, re) of a long row of v by one warp;
// chunks of the same row combine through atomicMax on the parents and atomicOr
// on F_{k+1}, whose first setter of any bit claims v for the queue (the level
// goes to the planes when v is expanded, as everywhere).
template <typename Word>
__device__ __forceinline__ void pull_chunk(const BatchParams& p, const Word* Fc, Word* Fn, int knext, int v,
                                           long long rb, long long re, uint64_t need, int lane, Claims& cl,
                                           int* wq, int& nbuf) {
  const Bits found = resolve_row<Word, true>(p, Fc, v, rb, re, need, lane);
  bool claimed = false;
  if (lane == 0 && found) {
    const Bits old = atomic_or_word(&Fn[v], found);
    if (old == 0) {
      claimed = true;
      const long long dout = __ldg(&p.off[v + 1]) - __ldg(&p.off[v]);  // (a directed graph's out-row may be short)
      if (dout > kChunkEdges) push_chunks_cta(p, knext, cl, v, dout);
    }
  }
  warp_enqueue(p, knext, wq, nbuf, claimed, v, lane, false);
}

// The rows of a frontier of at most one CTA's threads, with the prefix sums of
// their lengths.  (Their starts and words are read again at each visit, from L1:
// 8 KB more shared memory per CTA takes enough L1 to slow the pull levels by 3 %.)
struct FlatRows {
  int u[kBBlock];
  int pref[kBBlock];
};

// Vertices of a warp that have roots to find, waiting to be 32.
template <typename Word>
struct Pending {
  int v[64];
  Word need[64];
};

template <typename Word>
__global__ void __launch_bounds__(kBBlock, 2) batch_kernel(BatchParams p) {
  Word* F[3] = {static_cast<Word*>(p.F[0]), static_cast<Word*>(p.F[1]), static_cast<Word*>(p.F[2])};
  Word* V = static_cast<Word*>(p.V);
  __shared__ Claims cl;
  __shared__ LevelCtr s_ctr;             // counters of the level to expand, fetched by thread 0 at the barrier before it
  __shared__ int row_list[kBWarps][32];  // pull: the lanes whose rows a packed step examines
  __shared__ union {
    FlatRows flat;                 // top-down: the rows of a small frontier
    Pending<Word> pend[kBWarps];   // pull
  } s_rows;
  FlatRows& flat = s_rows.flat;
  __shared__ int scan_warp[kBWarps + 1];
  const int tid = threadIdx.x, lane = tid & 31;
  unsigned long long bar_target = 0;
  if (tid == 0) {
    bar_target = bfsdev::barrier_base(p.bar, gridDim.x);
    claims_reset(cl);
  }
  const long long G = gridDim.x;
  const long long gtid = (long long)blockIdx.x * kBBlock + tid;
  const long long gthreads = G * kBBlock;
  const long long gwarps = G * kBWarps;
  const long long gwarp = blockIdx.x + (long long)(tid >> 5) * G;  // round-robin over CTAs
  const unsigned nblocks = gridDim.x;

  // init: scratch parents of the vertices that an arc enters to -1 (atomicMax
  // offers need a floor; entries are only read where V says the root reached the
  // vertex), bitsets to 0, counters to 0
  const int S4 = p.stride / 4;  // 2 to 16, a power of two
  const int s4 = __ffs(S4) - 1;
  const long long total = (long long)p.n << s4;
  for (long long i = gtid; i < total; i += gthreads) {
    const long long v = i >> s4;
    if (!((__ldg(&p.dead[v >> 5]) >> (v & 31)) & 1u)) reinterpret_cast<int4*>(p.sp)[i] = make_int4(-1, -1, -1, -1);
  }
  for (long long v = gtid; v < p.n; v += gthreads) {
    F[0][v] = 0;
    F[1][v] = 0;
    F[2][v] = 0;
    V[v] = 0;
  }
  if (blockIdx.x == 0 && tid < kCtrRing * (int)(sizeof(LevelCtr) / 8))
    reinterpret_cast<unsigned long long*>(p.ctr)[tid] = 0ull;
  if (!bfsdev::grid_barrier(p.bar, nblocks, bar_target, p.spin_limit, p.status)) return;

  // seed: root r sets bit r of its own vertex (roots may repeat)
  if (blockIdx.x == 0 && tid < p.k) {
    const int s = p.src[tid];
    const uint64_t bit = 1ull << tid;
    p.sp[(long long)s * p.stride + tid] = s;  // level 0 has no plane bits
    atomic_or_word(&V[s], bit);
    const Bits old = atomic_or_word(&F[0][s], bit);
    if (old == 0) {
      const unsigned pos = atomicAdd(&p.ctr[0].count, 1u);
      p.queue[0][pos] = s;
      const long long deg = __ldg(&p.off[s + 1]) - __ldg(&p.off[s]);
      if (deg > kChunkEdges) push_chunks(p, 0, s, deg);
    }
  }
  if (!bfsdev::grid_barrier(p.bar, nblocks, bar_target, p.spin_limit, p.status, FetchCtr{&p.ctr[0], &s_ctr})) return;

  int k = 0;
  unsigned prev_count = 0;
  uint64_t t_prev = 0;
  if (p.stats && blockIdx.x == 0 && tid == 0) t_prev = bfsdev::global_timer_ns();
  for (;; ++k) {
    const unsigned count = s_ctr.count;  // (the next fetch comes after this level's work and a CTA barrier)
    if (count == 0) break;
    const unsigned nchunks = s_ctr.chunks;
    const Word* Fc = F[k % 3];
    Word* Fn = F[(k + 1) % 3];
    const int32_t* Q = p.queue[k % 3];
    const int knext = k + 1;
    if (blockIdx.x == 0 && tid < (int)(sizeof(LevelCtr) / 8))
      reinterpret_cast<unsigned long long*>(&p.ctr[(k + 4) % kCtrRing])[tid] = 0ull;
    if (k >= 1) {  // clear F_{k-1} for reuse as F_{k+2}
      Word* clr = F[(k + 2) % 3];
      const unsigned pc = prev_count;
      if ((long long)pc * 8 < p.n) {
        const int32_t* PQ = p.queue[(k + 2) % 3];
        for (long long i = gtid; i < pc; i += gthreads) clr[PQ[i]] = 0;
      } else {
        for (long long v = gtid; v < p.n; v += gthreads) clr[v] = 0;
      }
    }

    // the first level with bit j is 2^j: its plane is cleared one phase earlier
    if (((k + 1) & k) == 0) {
      Word* fresh = static_cast<Word*>(p.planes) + (long long)(31 - __clz(k + 1)) * p.n;
      for (long long v = gtid; v < p.n; v += gthreads) fresh[v] = 0;
    }

    const bool topdown = (long long)count <= p.td_limit;
    const int wid = tid >> 5;
    // A small frontier with few edges (the roots' own level, a traversal's tail):
    // every CTA takes in all its rows and edge i goes to thread i of the grid.  A
    // warp per row walked rows of up to kChunkEdges entries 32 at a time (17 roots
    // at scale 19: 18 us for the roots' level, 64 at scale 24: 105 us).
    int flat_total = INT_MAX;
    if (topdown && count <= (unsigned)kBBlock) {
      int u = -1, deg = 0, at = 0;
      if (tid < (int)count) {
        u = Q[tid];
        deg = (int)min((long long)__ldg(&p.off[u + 1]) - __ldg(&p.off[u]), 1ll << 21);  // the sum stays below 2^31
      }
      const int total = block_exclusive_scan(deg, scan_warp, at);
      if (total <= min(8 * gthreads, (1ll << 21) - 1)) {  // (no length was cut)
        flat_total = total;
        flat.u[tid] = u;
        flat.pref[tid] = at;
        if (u >= 0 && (unsigned)tid % nblocks == blockIdx.x) {
          const Bits f = (Bits)Fc[u];
          V[u] = (Word)((Bits)V[u] | f);
          add_level<Word>(p, u, f, k);
        }
        __syncthreads();
      }
    }
    if (flat_total != INT_MAX) {
      int room = kQBuf / kBBlock;  // steps that the CTA's claim buffer is sure to hold
      for (long long base = (long long)blockIdx.x * kBBlock; base < flat_total; base += gthreads) {
        if (room-- == 0) {
          flush_claims_if_full(p, knext, cl, kBBlock, kBigBuf / 2);
          room = 0;
        }
        const int idx = (int)base + tid;
        if (idx < flat_total) {
          int lo = 0, hi = kBBlock;  // the last row whose prefix sum is at most idx
          while (hi - lo > 1) {
            const int mid = (lo + hi) >> 1;
            if (flat.pref[mid] <= idx) lo = mid;
            else hi = mid;
          }
          const int u = flat.u[lo];
          const int w = __ldg(&p.adj[__ldg(&p.off[u]) + (idx - flat.pref[lo])]);
          td_visit(p, Fc, Fn, V, knext, (Bits)Fc[u], u, w, cl);
        }
      }
    } else if (topdown) {
      // frontier rows above kChunkEdges: one CTA per chunk item, with room in the
      // CTA's buffers for the item's claims
      const int64_t* items = p.chunks[k & 1];
      for (long long ci = blockIdx.x; ci < nchunks; ci += G) {
        flush_claims_if_full(p, knext, cl, kChunkEdges, kBigBuf / 2);
        const int64_t it = items[ci];
        const int u = (int)(it >> 32);
        const long long rb = __ldg(&p.off[u]) + (it & 0xffffffffll) * kChunkEdges;
        const long long re = min(rb + (long long)kChunkEdges, (long long)__ldg(&p.off[u + 1]));
        const uint64_t f = (Bits)Fc[u];
        for (long long j = rb + tid; j < re; j += kBBlock) td_visit(p, Fc, Fn, V, knext, f, u, __ldg(&p.adj[j]), cl);
      }
      // other frontier rows: one warp each; every frontier vertex folds its bits into V
      for (long long i = gwarp; i < count; i += gwarps) {
        const int u = Q[i];
        const uint64_t f = (Bits)Fc[u];
        if (lane == 0) {
          V[u] = (Word)((Bits)V[u] | f);
          add_level<Word>(p, u, f, k);
        }
        const long long b = __ldg(&p.off[u]), e = __ldg(&p.off[u + 1]);
        if (e - b > kChunkEdges) continue;
        for (long long j = b + lane; j < e; j += 32) td_visit(p, Fc, Fn, V, knext, f, u, __ldg(&p.adj[j]), cl);
      }
    } else {
      int* wq = cl.wq[wid];
      int nbuf = 0;
      // long rows: one warp per chunk of the static table
      for (long long ci = gwarp; ci < p.nbig; ci += gwarps) {
        const int64_t it = p.big[ci];
        const int v = (int)(it >> 32);
        const uint64_t need = __shfl_sync(kFull, ~((Bits)V[v] | (Bits)Fc[v]) & p.mask, 0);
        if (!need) continue;
        const long long rb = __ldg(&p.toff[v]) + (it & 0xffffffffll) * kChunkEdges;
        const long long re = min(rb + (long long)kChunkEdges, (long long)__ldg(&p.toff[v + 1]));
        pull_chunk(p, Fc, Fn, knext, v, rb, re, need, lane, cl, wq, nbuf);
      }
      // other rows: 32 vertices per warp; the owner lane updates V and F_{k+1}
      // word indices fit 32 bits: n < 2^31
      const int nw = (int)(((long long)p.n + 31) / 32), gw = (int)gwarps;
      constexpr int kGroupWords = 16;
      // words [0, S) are dealt one at a time round robin (warp i takes i, i + gw, ...),
      // the rest in groups of kGroupWords words from the level's cursor, each fetch issued
      // one group ahead.  Full row scans make some words far dearer than others: with an
      // all-static deal a level waited on its slowest warps (64 roots at R-MAT scale 26:
      // 104.6 ms, 94.4 with the dynamic tail).  With few words per warp all are dealt
      // round robin: 16-word groups from the first word left warps idle on the 2^27-edge
      // edgefactor-16 and -64 graphs (16 roots: 3 % and 4 % slower).
      const int S = nw > 64 * gw ? gw * ((nw / 2) / gw) : nw;
      const int ngroups = (nw - S + kGroupWords - 1) / kGroupWords;
      int* list = row_list[wid];
      // the warp's words in turn: ww, then next_word(ww), until nw
      unsigned fetched = 0;  // lane 0: the next group, fetched while the one before is worked on
      int wend = 0;
      if (ngroups > 0 && lane == 0) fetched = (unsigned)atomicAdd(&p.ctr[k % kCtrRing].pad, 1ull);
      auto take_group = [&]() {
        const int grp = (int)__shfl_sync(kFull, fetched, 0);
        if (grp >= ngroups) return nw;
        if (lane == 0) fetched = (unsigned)atomicAdd(&p.ctr[k % kCtrRing].pad, 1ull);
        wend = min(nw, S + (grp + 1) * kGroupWords);
        return S + grp * kGroupWords;
      };
      auto next_word = [&](int ww) {
        const int w1 = ww < S ? ww + gw : ww + 1;
        return w1 < (ww < S ? S : wend) ? w1 : take_group();
      };
      // A warp goes through its words, folds F_k into V and collects the vertices
      // that have roots to find; 32 of them at a time are resolved, one per lane, so
      // that a step's lanes and loads are filled however few of a word's vertices
      // are left (word by word a late level cost a chain of dependent loads for one
      // vertex: 64 roots at scale 24, level 5: 450 us).
      Pending<Word>& pend = s_rows.pend[wid];
      int npend = 0;
      for (int ww = (int)gwarp < S ? (int)gwarp : take_group();;) {
        const bool more = ww < nw;
        if (more) {
          const int v = ww * 32 + lane;  // (n rounded up to 32 fits: n < 2^31 - 1)
          const uint32_t dead = __ldg(&p.dead[ww]);  // the bits past n are set
          Bits need = 0;
          if (!((dead >> lane) & 1u)) {
            const Bits vv = (Bits)V[v], fv = (Bits)Fc[v];
            need = ~(vv | fv) & p.mask;
            if (fv) {
              V[v] = (Word)(vv | fv);
              add_level<Word>(p, v, fv, k);
            }
          } else if (v < p.n) {  // only a root can be here: no arc enters v
            const Bits fv = (Bits)Fc[v];
            if (fv) {
              V[v] = (Word)((Bits)V[v] | fv);
              add_level<Word>(p, v, fv, k);
            }
          }
          const unsigned m = __ballot_sync(kFull, need != 0);
          if (need) {
            const int at = npend + __popc(m & bfsdev::lanemask_lt());
            pend.v[at] = v;
            pend.need[at] = (Word)need;
          }
          npend += __popc(m);
          __syncwarp();
          ww = next_word(ww);
        }
        if (npend >= 32 || (!more && npend > 0)) {
          const int take = min(32, npend);
          npend -= take;
          int v = 0, deg = 0;
          long long e = 0;
          Bits need = 0;
          if (lane < take) {
            v = pend.v[npend + lane];
            e = __ldg(&p.toff[v + 1]);
            const long long d = e - __ldg(&p.toff[v]);
            if (d <= kChunkEdges) {  // (longer rows went by chunks above)
              deg = (int)d;
              need = (Bits)pend.need[npend + lane];
            }
          }
          __syncwarp();  // the entries are taken before the next word adds its own
          const Bits found = resolve_group(p, Fc, v, deg, e, need, lane, list);
          if (found) {
            Fn[v] = (Word)found;
            if (p.directed) {  // the next level's top-down expansion needs the chunks of a long out-row
              const long long dout = __ldg(&p.off[v + 1]) - __ldg(&p.off[v]);
              if (dout > kChunkEdges) push_chunks_cta(p, knext, cl, v, dout);
            }
          }
          warp_enqueue(p, knext, wq, nbuf, found != 0, v, lane, false);
        } else if (!more) {
          break;
        }
      }
      warp_enqueue(p, knext, wq, nbuf, false, 0, lane, true);
    }
    flush_claims(p, knext, cl);
    if (!bfsdev::grid_barrier(p.bar, nblocks, bar_target, p.spin_limit, p.status,
                              FetchCtr{&p.ctr[(k + 1) % kCtrRing], &s_ctr}))
      return;
    prev_count = count;
    if (p.stats && blockIdx.x == 0 && tid == 0 && k < kMaxStatLevels) {
      const uint64_t t = bfsdev::global_timer_ns();
      bfs_level_stat st{};
      st.frontier_count = count;
      st.time_ns = (int64_t)(t - t_prev);
      st.variant = topdown ? BFS_VARIANT_TD_WARP : BFS_VARIANT_PULL;
      p.stats[k] = st;
      t_prev = t;
    }
  }
  if (gtid == 0) p.misc[1] = k;

  // Outputs, root-major, from the scratch rows and planes (the loop ended right
  // after a grid barrier, so both are final, and V holds every root bit of every
  // vertex reached).  A warp takes 32 vertices, lane i the i-th: it reads its
  // scratch row 16 bytes at a time (skipped where none of the four roots reached
  // it), puts the levels together from the planes, and each root's 32 results
  // leave as one 128-byte store.  No CTA barrier, and four row loads in flight
  // per lane: through shared-memory tiles of 32 vertices per CTA the phase took
  // 5.4 ms for 64 roots at R-MAT scale 24.
  const int nplanes = k > 1 ? 32 - __clz(k - 1) : 0;  // levels 0 .. k - 1
  const Word* planes = static_cast<const Word*>(p.planes);
  constexpr int kRegPlanes = 3;
  const int ngroups = (p.k + 3) / 4;
  const long long ntiles = ((long long)p.n + 31) / 32;
  for (long long t = gwarp; t < ntiles; t += gwarps) {
    const long long v = t * 32 + lane;
    const bool in = v < p.n;
    const Bits vv = in ? (Bits)V[v] : 0ull;
    Bits pl[kRegPlanes];
#pragma unroll
    for (int j = 0; j < kRegPlanes; ++j) pl[j] = vv && j < nplanes ? (Bits)planes[(long long)j * p.n + v] : 0ull;
    const int4* row = reinterpret_cast<const int4*>(p.sp) + (v << s4);
#pragma unroll 4
    for (int c = 0; c < ngroups; ++c) {
      const unsigned on = (unsigned)(vv >> (4 * c)) & 15u;
      int4 pv = make_int4(-1, -1, -1, -1);
      if (on) pv = __ldcg(row + c);  // this launch wrote the rows, so not __ldg; used once, so from L2
      unsigned lb[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) lb[q] = 0;
#pragma unroll
      for (int j = 0; j < kRegPlanes; ++j) {
        const unsigned b = (unsigned)(pl[j] >> (4 * c));
#pragma unroll
        for (int q = 0; q < 4; ++q) lb[q] |= (b >> q & 1u) << j;
      }
      for (int j = kRegPlanes; j < nplanes; ++j) {
        const unsigned b = on ? (unsigned)((Bits)planes[(long long)j * p.n + v] >> (4 * c)) : 0u;
#pragma unroll
        for (int q = 0; q < 4; ++q) lb[q] |= (b >> q & 1u) << j;
      }
      const int pq[4] = {pv.x, pv.y, pv.z, pv.w};
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int r = 4 * c + q;
        if (r < p.k && in) {
          const bool reached = (on >> q) & 1u;
          p.level[(long long)r * p.n + v] = reached ? (int)lb[q] : -1;
          p.parent[(long long)r * p.n + v] = reached ? pq[q] : -1;
        }
      }
    }
  }
}

}  // namespace

int launch_batch(const BatchRequest& r, cudaStream_t s) {
  bfs_graph* g = r.g;
  Workspace* w = r.w;
  DeviceInfo di;
  if (int e = current_device_info(&di)) return e;
  if (r.width != 8 && r.width != 16 && r.width != 32 && r.width != 64)
    return fail(BFS_ERR_INVALID_ARG, "batch width must be 8, 16, 32 or 64");
  if (r.k < 1 || r.k > r.width) return fail(BFS_ERR_INVALID_ARG, "batch of 1..width roots expected");
  if (!g->d_off || !g->d_toff || (g->nnz > 0 && (!g->d_adj || !g->d_tadj)))
    return fail(BFS_ERR_INVALID_ARG, "graph without rows");
  if (int e = ensure_batch_state(g, w)) return e;
  const bfs_tuning t = effective_tuning(g);
  BatchParams p{};
  p.off = g->d_off;
  p.adj = g->d_adj;
  p.toff = g->d_toff;
  p.tadj = g->d_tadj;
  p.directed = g->directed ? 1 : 0;
  p.n = g->n;
  p.nnz = g->nnz;
  p.k = r.k;
  p.mask = r.k == 64 ? ~0ull : ((1ull << r.k) - 1ull);
  for (int i = 0; i < r.k; ++i) p.src[i] = r.h_sources[i];
  p.level = r.level;
  p.parent = r.parent;
  p.stride = r.width;
  p.sp = w->bscr;
  p.planes = w->bscr + (size_t)g->n * 64;
  p.dead = g->d_dead;
  for (int i = 0; i < 3; ++i) {
    p.F[i] = w->bset[i];
    p.queue[i] = w->queue[i];
  }
  p.V = w->bvis;
  p.chunks[0] = w->chunks[0];
  p.chunks[1] = w->chunks[1];
  p.chunk_cap = w->chunk_cap;
  p.big = g->d_big;
  p.nbig = g->nbig;
  p.ctr = w->ctr;
  p.status = w->status;
  p.misc = w->misc;
  p.stats = r.want_stats ? w->stats : nullptr;
  p.spin_limit = r.spin_limit ? r.spin_limit : (1u << 25);
  p.td_limit = t.batch_topdown_limit;
  const void* fn = r.width == 8    ? (const void*)batch_kernel<uint8_t>
                   : r.width == 16 ? (const void*)batch_kernel<uint16_t>
                   : r.width == 32 ? (const void*)batch_kernel<uint32_t>
                                   : (const void*)batch_kernel<uint64_t>;
  int per_sm = 0;
  BFS_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, kBBlock, 0));
  if (per_sm < 1) return fail(BFS_ERR_CUDA, "batch kernel cannot be resident");
  const int grid = per_sm * di.sm_count;
  if (int e = prepare_barrier(w, 1, grid, s, &p.bar)) return e;
  void* args[] = {&p};
  BFS_CUDA_TRY(cudaLaunchCooperativeKernel(fn, dim3(grid), dim3(kBBlock), args, 0, s));
  return BFS_OK;
}

}  // namespace bfsint
