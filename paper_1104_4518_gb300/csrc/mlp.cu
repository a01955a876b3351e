// The per-level variant selector network: forward pass, mean-squared-error
// gradient and Adam, on the device.  The network is 12 -> 64 -> 64 -> 4 with
// ReLU, float32 (layout in mlp_device.cuh).  Gradients are summed in a fixed
// order (per-tile partial sums, then a serial sum over tiles per parameter),
// so a training run is bit-reproducible.
#include <cmath>
#include <mutex>
#include <vector>

#include "internal.h"
#include "nvtx_range.h"
#include "mlp_device.cuh"

namespace bfsint {
namespace {

using namespace bfsdev;

constexpr int kFwdThreads = 128;
constexpr int kTS = 32;           // samples per gradient tile
constexpr int kGradThreads = 512;

__global__ void __launch_bounds__(kFwdThreads) mlp_forward_kernel(const float* __restrict__ params,
                                                                  const float* __restrict__ X, int B,
                                                                  float* __restrict__ Y) {
  extern __shared__ float s_w[];
  for (int i = threadIdx.x; i < BFS_MLP_PARAMS; i += kFwdThreads) s_w[i] = params[i];
  __syncthreads();
  const int s = blockIdx.x * kFwdThreads + threadIdx.x;
  if (s >= B) return;
  float x[12], h1[64], h2[64];
#pragma unroll
  for (int k = 0; k < 12; ++k) x[k] = X[(long long)s * 12 + k];
  for (int t = 0; t < 64; ++t) h1[t] = mlp_h1(s_w, x, t);
  for (int t = 0; t < 64; ++t) h2[t] = mlp_h2(s_w, h1, t);
#pragma unroll
  for (int o = 0; o < 4; ++o) Y[(long long)s * 4 + o] = mlp_out(s_w, h2, o);
}

constexpr int kW2Row = 68;  // padded row of W2 in shared memory: 16-byte loads along and across rows without conflicts

struct __align__(16) GradSmem {
  float w1[12 * 64], b1[64], b2[64], w3[64 * 4], b3[4];
  float w2[64 * kW2Row];
  float x[kTS][12];
  float h1[kTS][64];
  float h2[kTS][64];
  float dz1[kTS][64];
  float dz2[kTS][64];
  float dy[kTS][4];
  float sq[kTS * 4];  // squared errors by sample and output
};

// The reduction and the Adam step are launched to start while the kernel before
// them runs out (programmatic dependent launch): their CTAs take their places
// early and wait there for that kernel's end before they touch memory, which hides
// a launch's latency of about 2 us (1,379 samples: a gradient call 27.8 -> 25.7 us,
// a training step 22.5 -> 18.5).  What they read is not const __restrict__, as
// it may still be written when they start.
__device__ __forceinline__ void launch_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void wait_for_previous_kernel() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

template <typename... K, typename... A>
cudaError_t launch_early(void (*kernel)(K...), unsigned grid, unsigned block, cudaStream_t s, A... args) {
  cudaLaunchAttribute early[1];
  early[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  early[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(block);
  cfg.stream = s;
  cfg.attrs = early;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<K>(args)...);
}

// Partial gradient and squared error of one tile of kTS samples.  Thread
// (t, grp) computes unit t of four samples, so that a weight loaded from
// shared memory serves four products; the W2 gradient is 2 x 4 blocks in
// registers, the outputs 32 partial sums per warp.  Every sum keeps the order
// of the serial definitions (the forward pass's of mlp_device.cuh, samples
// ascending in the gradients).  1,379 samples: 22.6 us with one thread per
// output (two shared loads per product, 32-way bank conflicts down W2's
// columns, 256 serial additions of the loss), now 14 us, of which 10 are the chain of
// phases (ncu, cold caches).
__global__ void __launch_bounds__(kGradThreads) mlp_grad_tile_kernel(const float* __restrict__ params,
                                                                     const float* __restrict__ X,
                                                                     const float* __restrict__ T, int B,
                                                                     float* __restrict__ partial,
                                                                     float* __restrict__ partial_loss) {
  launch_dependents();
  extern __shared__ __align__(16) unsigned char s_raw[];
  GradSmem& g = *reinterpret_cast<GradSmem*>(s_raw);
  constexpr int kPer = kTS * 64 / kGradThreads;  // samples per thread: 4
  constexpr int kGrps = kGradThreads / 64;
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5, t = tid & 63, grp = tid >> 6;
  const long long s0 = (long long)blockIdx.x * kTS;
  for (int i = tid; i < 12 * 64; i += kGradThreads) g.w1[i] = params[kW1 + i];
#pragma unroll
  for (int i = 0; i < 1024 / kGradThreads; ++i) {
    const int q = i * kGradThreads + tid;  // 16-byte group q of W2
    const float* src = params + kW2 + 4 * q;
    float4 w;
    if ((reinterpret_cast<uintptr_t>(params) & 15u) == 0) w = *reinterpret_cast<const float4*>(src);
    else w = make_float4(src[0], src[1], src[2], src[3]);
    *reinterpret_cast<float4*>(&g.w2[(q >> 4) * kW2Row + 4 * (q & 15)]) = w;
  }
  if (tid < 256) g.w3[tid] = params[kW3 + tid];
  if (tid < 64) {
    g.b1[tid] = params[kB1 + tid];
    g.b2[tid] = params[kB2 + tid];
  }
  if (tid < 4) g.b3[tid] = params[kB3 + tid];
  for (int i = tid; i < kTS * 12; i += kGradThreads) {
    const int s = i / 12, k = i % 12;
    g.x[s][k] = (s0 + s < B) ? X[(s0 + s) * 12 + k] : 0.0f;
  }
  __syncthreads();
  {  // layer 1
    float a[kPer];
#pragma unroll
    for (int q = 0; q < kPer; ++q) a[q] = g.b1[t];
#pragma unroll
    for (int k = 0; k < 12; ++k) {
      const float w = g.w1[k * 64 + t];
#pragma unroll
      for (int q = 0; q < kPer; ++q) a[q] = fmaf(g.x[grp * kPer + q][k], w, a[q]);
    }
#pragma unroll
    for (int q = 0; q < kPer; ++q) g.h1[grp * kPer + q][t] = fmaxf(a[q], 0.0f);
  }
  __syncthreads();
  {  // layer 2: four partial dot products p0 .. p3 per unit, added as (p0 + p1) + (p2 + p3)
    float lo[kPer], hi[kPer];
#pragma unroll
    for (int q = 0; q < kPer; ++q) lo[q] = hi[q] = 0.0f;
#pragma unroll 1
    for (int r = 0; r < 4; ++r) {
      float a[kPer];
#pragma unroll
      for (int q = 0; q < kPer; ++q) a[q] = 0.0f;
#pragma unroll 2
      for (int i = 16 * r; i < 16 * r + 16; i += 4) {
        float w[4];
#pragma unroll
        for (int c = 0; c < 4; ++c) w[c] = g.w2[(i + c) * kW2Row + t];
#pragma unroll
        for (int q = 0; q < kPer; ++q) {
          const float4 h = *reinterpret_cast<const float4*>(&g.h1[grp * kPer + q][i]);
          a[q] = fmaf(h.x, w[0], a[q]);
          a[q] = fmaf(h.y, w[1], a[q]);
          a[q] = fmaf(h.z, w[2], a[q]);
          a[q] = fmaf(h.w, w[3], a[q]);
        }
      }
#pragma unroll
      for (int q = 0; q < kPer; ++q) {
        if (r < 2) lo[q] = r == 0 ? a[q] : lo[q] + a[q];
        else hi[q] = r == 2 ? a[q] : hi[q] + a[q];
      }
    }
#pragma unroll
    for (int q = 0; q < kPer; ++q) g.h2[grp * kPer + q][t] = fmaxf((lo[q] + hi[q]) + g.b2[t], 0.0f);
  }
  __syncthreads();
  const float scale = 2.0f / (4.0f * (float)B);
#pragma unroll
  for (int q = 0; q < kTS / (kGradThreads / 32); ++q) {  // outputs: one sample per warp and turn, lane = partial sum
    const int s = wid * (kTS / (kGradThreads / 32)) + q;
    const float ha = g.h2[s][lane], hb = g.h2[s][lane + 32];
#pragma unroll
    for (int o = 0; o < 4; ++o) {
      float v = fmaf(hb, g.w3[(lane + 32) * 4 + o], ha * g.w3[lane * 4 + o]);
#pragma unroll
      for (int m = 16; m >= 1; m >>= 1) v = v + __shfl_xor_sync(0xffffffffu, v, m);
      if (lane == o) {
        float d = 0.0f, sq = 0.0f;
        if (s0 + s < B) {
          const float diff = (v + g.b3[o]) - T[(s0 + s) * 4 + o];
          sq = diff * diff;
          d = scale * diff;
        }
        g.dy[s][o] = d;
        g.sq[s * 4 + o] = sq;
      }
    }
  }
  __syncthreads();
  {  // dz2 = (dy W3^T) * [h2 > 0]
    const float4 w = *reinterpret_cast<const float4*>(&g.w3[t * 4]);
#pragma unroll
    for (int q = 0; q < kPer; ++q) {
      const int s = grp * kPer + q;
      const float4 d = *reinterpret_cast<const float4*>(g.dy[s]);
      float a = fmaf(d.x, w.x, 0.0f);
      a = fmaf(d.y, w.y, a);
      a = fmaf(d.z, w.z, a);
      a = fmaf(d.w, w.w, a);
      g.dz2[s][t] = g.h2[s][t] > 0.0f ? a : 0.0f;
    }
  }
  __syncthreads();
  {  // dz1 = (dz2 W2^T) * [h1 > 0]
    float a[kPer];
#pragma unroll
    for (int q = 0; q < kPer; ++q) a[q] = 0.0f;
#pragma unroll 2
    for (int j = 0; j < 64; j += 4) {
      const float4 w = *reinterpret_cast<const float4*>(&g.w2[t * kW2Row + j]);
#pragma unroll
      for (int q = 0; q < kPer; ++q) {
        const float4 d = *reinterpret_cast<const float4*>(&g.dz2[grp * kPer + q][j]);
        a[q] = fmaf(d.x, w.x, a[q]);
        a[q] = fmaf(d.y, w.y, a[q]);
        a[q] = fmaf(d.z, w.z, a[q]);
        a[q] = fmaf(d.w, w.w, a[q]);
      }
    }
#pragma unroll
    for (int q = 0; q < kPer; ++q) {
      const int s = grp * kPer + q;
      g.dz1[s][t] = g.h1[s][t] > 0.0f ? a[q] : 0.0f;
    }
  }
  __syncthreads();
  float* out = partial + (long long)blockIdx.x * BFS_MLP_PARAMS;
  {  // W2: rows 2 ib and 2 ib + 1, columns 4 tb .. + 3
    const int ib = tid >> 4, tb = tid & 15;
    float a[2][4] = {};
#pragma unroll 4
    for (int s = 0; s < kTS; ++s) {
      const float2 h = *reinterpret_cast<const float2*>(&g.h1[s][2 * ib]);
      const float4 d = *reinterpret_cast<const float4*>(&g.dz2[s][4 * tb]);
      const float hv[2] = {h.x, h.y}, dv[4] = {d.x, d.y, d.z, d.w};
#pragma unroll
      for (int r = 0; r < 2; ++r)
#pragma unroll
        for (int c = 0; c < 4; ++c) a[r][c] = fmaf(hv[r], dv[c], a[r][c]);
    }
#pragma unroll
    for (int r = 0; r < 2; ++r)
      *reinterpret_cast<float4*>(out + kW2 + (2 * ib + r) * 64 + 4 * tb) = make_float4(a[r][0], a[r][1], a[r][2], a[r][3]);
  }
  {  // W1 at column t: row grp, and rows 8 + grp of the first four groups; W3 by the other four
    const bool first = grp < kGrps / 2;
    const int j = (tid - kGradThreads / 2) >> 2, o = tid & 3;
    float a = 0.0f, a2 = 0.0f;
#pragma unroll 4
    for (int s = 0; s < kTS; ++s) {
      const float d = g.dz1[s][t];
      a = fmaf(g.x[s][grp], d, a);
      a2 = first ? fmaf(g.x[s][kGrps + grp], d, a2) : fmaf(g.h2[s][j], g.dy[s][o], a2);
    }
    out[kW1 + grp * 64 + t] = a;
    if (first) out[kW1 + (kGrps + grp) * 64 + t] = a2;
    else out[kW3 + tid - kGradThreads / 2] = a2;
  }
  // biases and the tile's squared error, one kind per warp pair
  if (grp < 2) {
    float a = 0.0f;
#pragma unroll 8
    for (int s = 0; s < kTS; ++s) a += grp == 0 ? g.dz1[s][t] : g.dz2[s][t];
    out[(grp == 0 ? kB1 : kB2) + t] = a;
  } else if (grp == 2) {
    if (t < 4) {
      float a = 0.0f;
#pragma unroll 8
      for (int s = 0; s < kTS; ++s) a += g.dy[s][t];
      out[kB3 + t] = a;
    }
  } else if (t == 0) {
    float tot = 0.0f;
#pragma unroll 8
    for (int i = 0; i < kTS * 4; i += 4) {
      const float4 v = *reinterpret_cast<const float4*>(&g.sq[i]);
      tot += v.x;
      tot += v.y;
      tot += v.z;
      tot += v.w;
    }
    partial_loss[blockIdx.x] = tot;
  }
}
static_assert(kTS == 32 && kGradThreads == 512, "the gradient tile's thread mapping");

// Sums over the tiles, ascending: one thread per parameter, 16 loads in flight,
// and one for the loss.
__global__ void mlp_reduce_kernel(const float* partial, const float* partial_loss,
                                  int ntiles, int B, float* __restrict__ grad, float* __restrict__ loss) {
  launch_dependents();
  wait_for_previous_kernel();
  const int pidx = blockIdx.x * blockDim.x + threadIdx.x;
  if (pidx > BFS_MLP_PARAMS || (pidx == BFS_MLP_PARAMS && !loss)) return;
  const bool is_loss = pidx == BFS_MLP_PARAMS;
  const float* src = is_loss ? partial_loss : partial + pidx;
  const long long step = is_loss ? 1 : BFS_MLP_PARAMS;
  float a = 0.0f;
  int b = 0;
  for (; b + 16 <= ntiles; b += 16) {
    float v[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) v[i] = src[(b + i) * step];
#pragma unroll
    for (int i = 0; i < 16; ++i) a += v[i];
  }
  {
    float v[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) v[i] = b + i < ntiles ? src[(b + i) * step] : 0.0f;
#pragma unroll
    for (int i = 0; i < 16; ++i)
      if (b + i < ntiles) a += v[i];
  }
  if (is_loss) *loss = a / (4.0f * (float)B);
  else grad[pidx] = a;
}

__global__ void adam_kernel(float* __restrict__ params, const float* grad, float* __restrict__ m,
                            float* __restrict__ v, float lr, float beta1, float beta2, float eps, float bc1,
                            float bc2) {
  wait_for_previous_kernel();
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= BFS_MLP_PARAMS) return;
  const float gi = grad[i];
  const float mi = beta1 * m[i] + (1.0f - beta1) * gi;
  const float vi = beta2 * v[i] + (1.0f - beta2) * gi * gi;
  m[i] = mi;
  v[i] = vi;
  const float mhat = mi / bc1;
  const float vhat = vi / bc2;
  params[i] -= lr * mhat / (sqrtf(vhat) + eps);
}

size_t grad_smem_bytes() { return sizeof(GradSmem); }

int grad_impl(const float* params, const float* X, const float* T, int B, float* grad, float* loss,
              float* partial, float* partial_loss, cudaStream_t s) {
  const int ntiles = (B + kTS - 1) / kTS;
  static bool configured = false;
  if (!configured) {
    BFS_CUDA_TRY(cudaFuncSetAttribute(mlp_grad_tile_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      (int)grad_smem_bytes()));
    configured = true;
  }
  mlp_grad_tile_kernel<<<ntiles, kGradThreads, grad_smem_bytes(), s>>>(params, X, T, B, partial, partial_loss);
  BFS_CUDA_TRY(cudaGetLastError());
  BFS_CUDA_TRY(launch_early(mlp_reduce_kernel, BFS_MLP_PARAMS / 64 + 1, 64, s, partial, partial_loss, ntiles, B, grad, loss));
  return BFS_OK;
}

// ---------------- selector parameters of this process ----------------
std::mutex g_sel_mu;
std::vector<float> g_sel_host;
std::vector<float*> g_sel_dev;  // per device ordinal

}  // namespace

const float* learned_params_device(cudaStream_t s) {
  std::lock_guard<std::mutex> lk(g_sel_mu);
  if (g_sel_host.empty()) return nullptr;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return nullptr;
  if ((int)g_sel_dev.size() <= dev) g_sel_dev.resize(dev + 1, nullptr);
  if (!g_sel_dev[dev]) {
    std::vector<float> warp(BFS_MLP_PARAMS);
    for (int i = 0; i < BFS_MLP_PARAMS; ++i) warp[bfsdev::warp_layout_index(i)] = g_sel_host[i];
    float* p = nullptr;
    if (dev_alloc((void**)&p, sizeof(float) * BFS_MLP_PARAMS, "selector parameters") != BFS_OK) return nullptr;
    // there before any stream reads them: a pageable copy may still be on its way when the call returns
    SetupStream setup(s);
    if (setup.status() != cudaSuccess ||
        cudaMemcpyAsync(p, warp.data(), sizeof(float) * BFS_MLP_PARAMS, cudaMemcpyHostToDevice, setup) != cudaSuccess ||
        setup.done(true) != cudaSuccess) {
      dev_free(p);
      return nullptr;
    }
    g_sel_dev[dev] = p;
  }
  return g_sel_dev[dev];
}

void graph_feature_constants(int32_t n, int64_t nnz, float* log_n, float* log_nnz, float* inv_n, float* inv_nnz) {
  const float fn = (float)(n > 1 ? n : 1);
  const float fe = (float)(nnz > 1 ? nnz : 1);
  *log_n = log2f(fn) * 0.03125f;
  *log_nnz = log2f(fe) * 0.03125f;
  *inv_n = 1.0f / fn;
  *inv_nnz = 1.0f / fe;
}

}  // namespace bfsint

using namespace bfsint;

extern "C" {

int bfs_mlp_forward(const float* params, const float* X, int32_t B, float* Y, void* stream) {
  if (!params || !X || !Y || B < 0) return fail(BFS_ERR_INVALID_ARG, "bfs_mlp_forward: bad argument");
  if (B == 0) return BFS_OK;
  cudaStream_t s = (cudaStream_t)stream;
  static bool configured = false;
  if (!configured) {
    BFS_CUDA_TRY(cudaFuncSetAttribute(mlp_forward_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      (int)(sizeof(float) * BFS_MLP_PARAMS)));
    configured = true;
  }
  mlp_forward_kernel<<<(B + kFwdThreads - 1) / kFwdThreads, kFwdThreads, sizeof(float) * BFS_MLP_PARAMS, s>>>(
      params, X, B, Y);
  BFS_CUDA_TRY(cudaGetLastError());
  return BFS_OK;
}

int bfs_mlp_loss_grad(const float* params, const float* X, const float* T, int32_t B, float* grad, float* loss,
                      void* stream) {
  if (!params || !X || !T || !grad || B < 1) return fail(BFS_ERR_INVALID_ARG, "bfs_mlp_loss_grad: bad argument");
  cudaStream_t s = (cudaStream_t)stream;
  const int ntiles = (B + kTS - 1) / kTS;
  float* partial = nullptr;
  if (int e = dev_alloc((void**)&partial, sizeof(float) * ((size_t)ntiles * BFS_MLP_PARAMS + ntiles), "MLP partials"))
    return e;
  int rc = grad_impl(params, X, T, B, grad, loss, partial, partial + (size_t)ntiles * BFS_MLP_PARAMS, s);
  cudaError_t err = cudaStreamSynchronize(s);
  dev_free(partial);
  if (rc) return rc;
  if (err != cudaSuccess) return cuda_fail(err, "bfs_mlp_loss_grad");
  return BFS_OK;
}

int bfs_mlp_adam(float* params, const float* grad, float* m, float* v, int32_t t, float lr, float beta1, float beta2,
                 float eps, void* stream) {
  if (!params || !grad || !m || !v || t < 1) return fail(BFS_ERR_INVALID_ARG, "bfs_mlp_adam: bad argument");
  const float bc1 = (float)(1.0 - std::pow((double)beta1, (double)t));
  const float bc2 = (float)(1.0 - std::pow((double)beta2, (double)t));
  BFS_CUDA_TRY(launch_early(adam_kernel, (BFS_MLP_PARAMS + 255) / 256, 256, (cudaStream_t)stream, params, grad, m, v, lr,
                            beta1, beta2, eps, bc1, bc2));
  return BFS_OK;
}

int bfs_selector_train(float* params, const float* X, const float* T, int32_t B, int32_t steps, float lr,
                       float* loss_history, void* stream) {
  NvtxRange nvtx_range("bfs_selector_train");
  if (!params || !X || !T || B < 1 || steps < 0) return fail(BFS_ERR_INVALID_ARG, "bfs_selector_train: bad argument");
  cudaStream_t s = (cudaStream_t)stream;
  const int ntiles = (B + kTS - 1) / kTS;
  float* buf = nullptr;
  const size_t nfl = (size_t)ntiles * BFS_MLP_PARAMS + ntiles + 3 * (size_t)BFS_MLP_PARAMS;
  if (int e = dev_alloc((void**)&buf, sizeof(float) * nfl, "training buffers")) return e;
  float* partial = buf;
  float* ploss = partial + (size_t)ntiles * BFS_MLP_PARAMS;
  float* grad = ploss + ntiles;
  float* m = grad + BFS_MLP_PARAMS;
  float* v = m + BFS_MLP_PARAMS;
  int rc = BFS_OK;
  cudaError_t err = cudaMemsetAsync(m, 0, sizeof(float) * 2 * BFS_MLP_PARAMS, s);
  if (err != cudaSuccess) rc = cuda_fail(err, "memset");
  for (int t = 1; rc == BFS_OK && t <= steps; ++t) {
    rc = grad_impl(params, X, T, B, grad, loss_history ? loss_history + (t - 1) : nullptr, partial, ploss, s);
    if (rc == BFS_OK) rc = bfs_mlp_adam(params, grad, m, v, t, lr, 0.9f, 0.999f, 1e-8f, stream);
  }
  err = cudaStreamSynchronize(s);
  dev_free(buf);
  if (rc) return rc;
  if (err != cudaSuccess) return cuda_fail(err, "bfs_selector_train");
  return BFS_OK;
}

int bfs_selector_set_params(const float* params) {
  std::lock_guard<std::mutex> lk(g_sel_mu);
  for (float* p : g_sel_dev)
    if (p) dev_free(p);
  g_sel_dev.clear();
  if (!params) {
    g_sel_host.clear();
    return BFS_OK;
  }
  g_sel_host.assign(params, params + BFS_MLP_PARAMS);
  return BFS_OK;
}

int bfs_selector_load(const char* path) {
  if (!path) return fail(BFS_ERR_INVALID_ARG, "bfs_selector_load: NULL path");
  FILE* f = fopen(path, "rb");
  if (!f) return fail(BFS_ERR_INVALID_ARG, std::string("bfs_selector_load: cannot open ") + path);
  std::vector<float> w(BFS_MLP_PARAMS);
  const size_t got = fread(w.data(), sizeof(float), BFS_MLP_PARAMS, f);
  fclose(f);
  if (got != (size_t)BFS_MLP_PARAMS) return fail(BFS_ERR_INVALID_ARG, "bfs_selector_load: short file");
  return bfs_selector_set_params(w.data());
}

int bfs_selector_save(const char* path) {
  if (!path) return fail(BFS_ERR_INVALID_ARG, "bfs_selector_save: NULL path");
  std::vector<float> w;
  {
    std::lock_guard<std::mutex> lk(g_sel_mu);
    w = g_sel_host;
  }
  if (w.empty()) return fail(BFS_ERR_INVALID_ARG, "bfs_selector_save: no network set");
  FILE* f = fopen(path, "wb");
  if (!f) return fail(BFS_ERR_INVALID_ARG, std::string("bfs_selector_save: cannot open ") + path);
  const size_t put = fwrite(w.data(), sizeof(float), BFS_MLP_PARAMS, f);
  fclose(f);
  if (put != (size_t)BFS_MLP_PARAMS) return fail(BFS_ERR_INVALID_ARG, "bfs_selector_save: write failed");
  return BFS_OK;
}

int bfs_level_features(int32_t n, int64_t nnz, int32_t k, int64_t frontier_count, int64_t frontier_edges,
                       int64_t unvisited_count, int64_t unvisited_edges, const int64_t* bin_count, float* out12) {
  if (!bin_count || !out12) return fail(BFS_ERR_INVALID_ARG, "bfs_level_features: NULL pointer");
  // the float32 expressions of the in-loop selector (bfsdev::warp_level_features)
  float rn = 0.0f, re = 0.0f;
  bfsint::graph_feature_constants(n, nnz, &out12[0], &out12[1], &rn, &re);
  const float c = (float)frontier_count, d = (float)frontier_edges;
  const float rc = 1.0f / (frontier_count > 1 ? c : 1.0f);
  out12[2] = log2f(1.0f + (float)k) * 0.1f;
  out12[3] = log2f(1.0f + c) * 0.03125f;
  out12[4] = log2f(1.0f + d) * 0.03125f;
  out12[5] = c * rn;
  out12[6] = d * re;
  out12[7] = (float)unvisited_count * rn;
  out12[8] = (float)unvisited_edges * re;
  out12[9] = (float)bin_count[0] * rc;
  out12[10] = (float)bin_count[1] * rc;
  out12[11] = (float)bin_count[2] * rc;
  return BFS_OK;
}

}  // extern "C"
