// The selector network's forward pass.  The in-loop selector evaluates it with
// four warps (lane l computes hidden units l and l + 32 of each layer, the output
// layer as 32 partial sums combined by a butterfly of shuffles); the
// stand-alone kernels evaluate the same sums in the same association order,
// one thread per row, so both give bit-identical scores.
#pragma once

#include "bfs.h"

namespace bfsdev {

// Offsets of the parameter blocks in the flat vector:
// W1[12][64], b1[64], W2[64][64], b2[64], W3[64][4], b3[4].
constexpr int kW1 = 0;
constexpr int kB1 = kW1 + 12 * 64;
constexpr int kW2 = kB1 + 64;
constexpr int kB2 = kW2 + 64 * 64;
constexpr int kW3 = kB2 + 64;
constexpr int kB3 = kW3 + 64 * 4;
static_assert(kB3 + 4 == BFS_MLP_PARAMS, "parameter layout");

// Hidden unit t (< 64) of layer 1 for input x[12].
__device__ __forceinline__ float mlp_h1(const float* w, const float* x, int t) {
  float a = w[kB1 + t];
#pragma unroll
  for (int k = 0; k < 12; ++k) a = fmaf(x[k], w[kW1 + k * 64 + t], a);
  return fmaxf(a, 0.0f);
}

// Hidden unit t (< 64) of layer 2: four partial dot products over inputs
// 16r .. 16r+15 (r < 4), added as (p0 + p1) + (p2 + p3), then the bias.
__device__ __forceinline__ float mlp_h2(const float* w, const float* h1, int t) {
  float a[4];
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    a[r] = 0.0f;
#pragma unroll
    for (int i = 16 * r; i < 16 * r + 16; ++i) a[r] = fmaf(h1[i], w[kW2 + i * 64 + t], a[r]);
  }
  return fmaxf(((a[0] + a[1]) + (a[2] + a[3])) + w[kB2 + t], 0.0f);
}

// Partial sum j (< 32) of output o: inputs j (value hj) and j + 32 (value hj32).
__device__ __forceinline__ float mlp_out_part(const float* w, float hj, float hj32, int o, int j) {
  return fmaf(hj32, w[kW3 + (j + 32) * 4 + o], hj * w[kW3 + j * 4 + o]);
}

// Output o, one thread: the 32 partial sums combined pairwise at distance
// 16 .. 1 (the order of a shuffle butterfly over 32 lanes), then the bias.
__device__ __forceinline__ float mlp_out(const float* w, const float* h2, int o) {
  float p[32];
#pragma unroll
  for (int j = 0; j < 32; ++j) p[j] = mlp_out_part(w, h2[j], h2[j + 32], o, j);
#pragma unroll
  for (int m = 16; m >= 1; m >>= 1)
#pragma unroll
    for (int j = 0; j < m; ++j) p[j] = p[j] + p[j + m];
  return p[0] + w[kB3 + o];
}

// Exact float of a nonnegative 64-bit count.  Values below 2^32 go through the
// 32-bit conversion, which gives the same float and pipelines far better than
// the 64-bit one; the branch is uniform when every lane converts the same value.
__device__ __forceinline__ float count_to_float(long long v) {
  return ((unsigned long long)v >> 32) ? (float)v : (float)(unsigned)v;
}

// The 12 level features (see bfs_level_features in bfs.h), the same float32
// expressions as the host function, on a whole warp: lane l of the first ten
// computes feature l + 2 from its own count, so that the conversions, logarithms
// and products of all of them run once (one lane doing all twelve took 0.5 us of
// a level).  f0 = log2(n) / 32, f1 = log2(nnz) / 32, rn = 1 / n and re = 1 / nnz
// are constants of the graph, passed in; x is the same in every lane.
__device__ __forceinline__ void warp_level_features(float f0, float f1, float rn, float re, int k, long long count,
                                                    long long edges, long long unvisited, long long unvisited_edges,
                                                    const unsigned long long* bins, int lane, float (&x)[12]) {
  // each lane's count: k, c, d, c, d, unvisited, unvisited edges, bins
  long long mine = (lane & 1) ? count : edges;
  if (lane == 0) mine = k;
  if (lane == 5) mine = unvisited;
  if (lane == 6) mine = unvisited_edges;
  if (lane >= 7 && lane < 10) mine = (long long)bins[lane - 7];
  const float v = count_to_float(mine);
  const float c = __shfl_sync(0xffffffffu, v, 1);
  const float rc = 1.0f / (c > 1.0f ? c : 1.0f);
  float f;
  if (lane < 3) f = log2f(1.0f + v) * (lane == 0 ? 0.1f : 0.03125f);
  else f = v * (lane >= 7 ? rc : (lane & 1) ? rn : re);  // lanes 3, 5: over n; 4, 6: over nnz
  x[0] = f0;
  x[1] = f1;
#pragma unroll
  for (int i = 0; i < 10; ++i) x[i + 2] = __shfl_sync(0xffffffffu, f, i);
}

// ---- the network on four warps ----
// The in-loop selector keeps the parameters in shared memory in a layout for a
// warp: in the blocks W1, b1, W2, b2 (each made of rows of 64), entry t of a
// row moves to position 2 (t mod 32) + t / 32, so lane l reads the weights of
// its units l and l + 32 as one float2.  W3 and b3 keep their places (lane j
// reads W3 rows j and j + 32 as float4).  The arithmetic is that of mlp_h1,
// mlp_h2 and mlp_out, in the same order.
__host__ __device__ __forceinline__ int warp_layout_index(int i) {
  if (i >= kW3) return i;
  const int t = i & 63;
  return (i - t) + 2 * (t & 31) + (t >> 5);
}

// On the first four warps of a CTA: every warp computes layer 1 (in its own h1,
// so that none waits for another), warp r partial dot product r of layer 2, and
// warp o output o; mlp_argmin picks from the outputs after a CTA barrier.
struct __align__(16) MlpScratch {
  float h1[4][64];
  float part[4][64];
};
constexpr int kMlpThreads = 128;

// x: the 12 features (the same values in every lane); w: parameters in the warp
// layout; warp in [0, 4).  Each group of shared-memory loads is issued before
// the multiply-adds that use it, so their latencies overlap.  Uses named
// barrier 1.
__device__ __forceinline__ void warps_mlp_outputs(const float* __restrict__ w, const float* x, MlpScratch& sc, float* y_out,
                                                  int warp, int lane) {
  float* h1 = sc.h1[warp];
  {
    const float2 bias1 = reinterpret_cast<const float2*>(w + kB1)[lane];
    float2 w1[12];
#pragma unroll
    for (int k = 0; k < 12; ++k) w1[k] = reinterpret_cast<const float2*>(w + kW1 + k * 64)[lane];
    float a = bias1.x, c = bias1.y;
#pragma unroll
    for (int k = 0; k < 12; ++k) {
      a = fmaf(x[k], w1[k].x, a);
      c = fmaf(x[k], w1[k].y, c);
    }
    h1[lane] = fmaxf(a, 0.0f);
    h1[lane + 32] = fmaxf(c, 0.0f);
  }
  __syncwarp();
  {
    float2 wv[16];
    float hs[16];
#pragma unroll
    for (int e = 0; e < 16; ++e) wv[e] = reinterpret_cast<const float2*>(w + kW2 + (16 * warp + e) * 64)[lane];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const float4 hv = reinterpret_cast<const float4*>(h1)[4 * warp + q];
      hs[4 * q] = hv.x;
      hs[4 * q + 1] = hv.y;
      hs[4 * q + 2] = hv.z;
      hs[4 * q + 3] = hv.w;
    }
    float a = 0.0f, c = 0.0f;
#pragma unroll
    for (int e = 0; e < 16; ++e) {
      a = fmaf(hs[e], wv[e].x, a);
      c = fmaf(hs[e], wv[e].y, c);
    }
    sc.part[warp][lane] = a;
    sc.part[warp][lane + 32] = c;
  }
  const float2 bias2 = reinterpret_cast<const float2*>(w + kB2)[lane];
  const float w3a = w[kW3 + lane * 4 + warp], w3c = w[kW3 + (lane + 32) * 4 + warp], b3 = w[kB3 + warp];
  asm volatile("bar.sync 1, %0;" ::"n"(kMlpThreads) : "memory");
  const float h2a = fmaxf(((sc.part[0][lane] + sc.part[1][lane]) + (sc.part[2][lane] + sc.part[3][lane])) + bias2.x, 0.0f);
  const float h2c = fmaxf(((sc.part[0][lane + 32] + sc.part[1][lane + 32]) +
                           (sc.part[2][lane + 32] + sc.part[3][lane + 32])) + bias2.y, 0.0f);
  float y = fmaf(h2c, w3c, h2a * w3a);
#pragma unroll
  for (int m = 16; m >= 1; m >>= 1) y = y + __shfl_xor_sync(0xffffffffu, y, m);
  if (lane == 0) y_out[warp] = y + b3;
}

// The index of the smallest output.
__device__ __forceinline__ int mlp_argmin(const float4 y) {
  int best = 0;
  float yb = y.x;
  if (y.y < yb) best = 1, yb = y.y;
  if (y.z < yb) best = 2, yb = y.z;
  if (y.w < yb) best = 3;
  return best;
}

}  // namespace bfsdev
