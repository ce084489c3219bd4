// Learned warm start: training and stand-alone inference of the 16-64-64-3 network on the GPU.
// The network maps the 16 features of a contact to its (normal, t1, t2) impulses; it is trained
// on rows harvested from cold-start rollouts (features, converged impulses) by minimising the
// mean squared error. Forward and reverse passes run on the bfloat16 tensor cores with the
// storage points of the in-step inference (inputs, weights and hidden activations in bfloat16,
// fp32 accumulation, straight-through rounding in reverse mode); the weight gradient is the
// split-K reduction of the stored deltas against the stored activations (one launch for the three
// layers and their biases); Adam updates the fp32 master weights.
#include <cuda_runtime.h>

#include <algorithm>

#include "../../include/dp.h"
#include "dp_kernels.h"
#include "dp_mma.cuh"
#include "dp_world.h"

namespace {

constexpr int WS_ROW = 19;       // harvested row: 16 features, 3 impulses
constexpr int WS_WARPS = 4;      // warps per block of the row kernels
constexpr int ACT_ROWS = WsTC::K0 + WsTC::H1 + WsTC::H2;   // stored activations per row
constexpr int DEL_ROWS = WsTC::H1 + WsTC::H2 + WsTC::NO;   // stored deltas per row

// Flat fp32 parameters -> tensor-core layouts (zero padded) and the bias array.
__global__ void k_ws_prep(const float* __restrict__ W, __nv_bfloat16* tc, float* bias) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p < WsTC::BSIZE) {
    float v = 0.f;
    if (p < WsTC::B2) v = W[WsTC::F_B1 + p];
    else if (p < WsTC::B3) v = W[WsTC::F_B2 + p - WsTC::B2];
    else if (p - WsTC::B3 < WsTC::NO) v = W[WsTC::F_B3 + p - WsTC::B3];
    bias[p] = v;
  }
  if (p >= WsTC::SIZE) return;
  auto w1 = [&](int o, int i) { return W[WsTC::F_W1 + o * WsTC::K0 + i]; };
  auto w2 = [&](int o, int i) { return W[WsTC::F_W2 + o * WsTC::H1 + i]; };
  auto w3 = [&](int o, int i) { return o < WsTC::NO ? W[WsTC::F_W3 + o * WsTC::H2 + i] : 0.f; };
  float v;
  if (p < WsTC::W2) {  // W1 [64][16]
    v = w1(p / 16, p % 16);
  } else if (p < WsTC::W3) {  // W2 [64][64]
    const int q = p - WsTC::W2;
    v = w2(q / WsTC::H1, q % WsTC::H1);
  } else if (p < WsTC::W3T) {  // W3 [8][64]
    const int q = p - WsTC::W3;
    v = w3(q / WsTC::H2, q % WsTC::H2);
  } else if (p < WsTC::W2T) {  // W3^T [64][16]
    const int q = p - WsTC::W3T;
    v = w3(q % 16, q / 16);
  } else if (p < WsTC::W1T) {  // W2^T [64][64]
    const int q = p - WsTC::W2T;
    v = w2(q % WsTC::H2, q / WsTC::H2);
  } else {  // W1^T [16][64]
    const int q = p - WsTC::W1T;
    v = w1(q % WsTC::H1, q / WsTC::H1);
  }
  tc[p] = __float2bfloat16_rn(v);
}

// Inference: y[n][3] for features x[n][stride] (first 16 columns).
__global__ void __launch_bounds__(32 * WS_WARPS) k_ws_infer(const __nv_bfloat16* __restrict__ tc,
                                                             const float* __restrict__ bias,
                                                             const float* __restrict__ x, int stride, long long n,
                                                             float* __restrict__ y) {
  const long long base = ((long long)blockIdx.x * WS_WARPS + (threadIdx.x >> 5)) * 32;
  if (base >= n) return;  // whole warp leaves together
  mlp3_forward<WsTC::K0, WsTC::H1, WsTC::H2, WsTC::NO>(
      WsTC::K0, WsTC::NO,
      [&](int f, int r) { return base + r < n ? x[(base + r) * stride + f] : 0.f; }, tc + WsTC::W1, bias + WsTC::B1,
      tc + WsTC::W2, bias + WsTC::B2, tc + WsTC::W3, bias + WsTC::B3,
      [&](int f, int r, float v) {
        if (base + r < n) y[(base + r) * WsTC::NO + f] = v;
      },
      [](int, int, int, float) {});
}

// Forward and reverse pass of the squared-error loss on 32 rows per warp. Stores, per row
// column (stride np = n rounded up to 32): act = [bf16 features (16), hidden 1 (64), hidden 2
// (64)], del = [delta hidden 1 (64), delta hidden 2 (64), delta output (3)], and the warp's
// partial sum of squared errors. Padded rows have zero deltas.
__global__ void __launch_bounds__(32 * WS_WARPS) k_ws_fwdbwd(const __nv_bfloat16* __restrict__ tc,
                                                              const float* __restrict__ bias,
                                                              const float* __restrict__ rows, long long n,
                                                              long long np, float inv_n, float* __restrict__ act,
                                                              float* __restrict__ del, float* __restrict__ loss_part) {
  __shared__ float ys[WS_WARPS][WsTC::NO][32];
  __shared__ float ubs[WS_WARPS][WsTC::NO][32];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const long long wid = (long long)blockIdx.x * WS_WARPS + warp;
  const long long base = wid * 32;
  if (base >= np) return;
  const long long me = base + lane;
  const bool valid = me < n;
  for (int f = 0; f < WsTC::K0; ++f) act[(size_t)f * np + me] = valid ? bf16r(rows[me * WS_ROW + f]) : 0.f;
  auto col = [&](int r) { return base + r; };
  mlp3_forward<WsTC::K0, WsTC::H1, WsTC::H2, WsTC::NO>(
      WsTC::K0, WsTC::NO,
      [&](int f, int r) { return col(r) < n ? rows[col(r) * WS_ROW + f] : 0.f; }, tc + WsTC::W1, bias + WsTC::B1,
      tc + WsTC::W2, bias + WsTC::B2, tc + WsTC::W3, bias + WsTC::B3,
      [&](int f, int r, float v) { ys[warp][f][r] = v; },
      [&](int l, int f, int r, float v) {
        act[(size_t)((l == 1 ? WsTC::K0 : WsTC::K0 + WsTC::H1) + f) * np + col(r)] = col(r) < n ? v : 0.f;
      });
  __syncwarp();
  float e = 0.f;
  for (int k = 0; k < WsTC::NO; ++k) {
    const float d = valid ? ys[warp][k][lane] - rows[me * WS_ROW + WsTC::K0 + k] : 0.f;
    e += d * d;
    const float g = 2.f * d * inv_n;
    ubs[warp][k][lane] = g;
    del[(size_t)(WsTC::H1 + WsTC::H2 + k) * np + me] = g;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) e += __shfl_xor_sync(0xffffffffu, e, o);
  if (lane == 0) loss_part[wid] = e;
  __syncwarp();
  mlp3_backward<WsTC::K0, WsTC::H1, WsTC::H2, WsTC::NO>(
      WsTC::K0, WsTC::NO,
      [&](int f, int r) { return ubs[warp][f][r]; }, tc + WsTC::W3T, tc + WsTC::W2T, tc + WsTC::W1T,
      [&](int l, int f, int r) {
        return act[(size_t)((l == 1 ? WsTC::K0 : WsTC::K0 + WsTC::H1) + f) * np + col(r)] > 0.f;
      },
      [&](int l, int f, int r, float v) { del[(size_t)((l == 1 ? 0 : WsTC::H1) + f) * np + col(r)] = v; },
      [](int, int, float) {});
}

// Split-K weight and bias gradient, all three layers in one launch (blockIdx.y: the layer, blockIdx.x:
// the split's columns): partial[split] holds a whole gradient in the master weights' layout. A CTA of
// 256 threads forms the layer's M x C products (M, C <= 64; up to 4 x 4 per thread, fp32) 32 columns at a
// time, the next columns on their way in registers meanwhile; thread t < M also sums delta row t, the
// bias gradient.
// Bound: FFMA (32768 rows: 0.35 GFLOP), if the chip is full. A split per
// 16384 columns left two CTAs on 152 SMs: 5634 us at 32768 rows. With one per 256 columns (at most
// 256) the three layers are 384 CTAs there: the whole training step 5673 -> 82 us, and 70 us with each
// layer's own tile (a 64 x 64 tile for all three kept 1.5 of 3 tiles' products for padding).
constexpr int DW_K = 32, DW_LD = DW_K + 4;
template <int M, int C>
__device__ __forceinline__ void ws_dw_layer(float (&As)[64][DW_LD], float (&Bs)[64][DW_LD], const float* __restrict__ dl,
                                            const float* __restrict__ al, long long np, long long chunk, float* __restrict__ W,
                                            float* __restrict__ b) {
  constexpr int U = (M + 15) / 16, V = (C + 15) / 16;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const long long n0 = (long long)blockIdx.x * chunk, n1 = min(np, n0 + chunk);  // multiples of DW_K
  const int tx = tid & 15, ty = tid >> 4;
  float ra[2 * U], rb[2 * V];
  auto fetch = [&](long long n) {  // a warp takes every eighth row of each operand, a lane one column
#pragma unroll
    for (int q = 0; q < 2 * U; ++q) ra[q] = warp + 8 * q < M ? __ldg(dl + (size_t)(warp + 8 * q) * np + n + lane) : 0.f;
#pragma unroll
    for (int q = 0; q < 2 * V; ++q) rb[q] = warp + 8 * q < C ? __ldg(al + (size_t)(warp + 8 * q) * np + n + lane) : 0.f;
  };
  float acc[U][V] = {}, bsum = 0.f;
  const bool work = ty < M && tx < C;  // rows ty + 16 u, columns tx + 16 v
  if (n0 < n1) fetch(n0);
  for (long long n = n0; n < n1; n += DW_K) {
#pragma unroll
    for (int q = 0; q < 2 * U; ++q) As[warp + 8 * q][lane] = ra[q];
#pragma unroll
    for (int q = 0; q < 2 * V; ++q) Bs[warp + 8 * q][lane] = rb[q];
    __syncthreads();
    if (n + DW_K < n1) fetch(n + DW_K);
    if (work) {
#pragma unroll
      for (int k = 0; k < DW_K; k += 4) {
        float4 x[U], y[V];
#pragma unroll
        for (int u = 0; u < U; ++u) x[u] = *reinterpret_cast<const float4*>(&As[ty + 16 * u][k]);
#pragma unroll
        for (int v = 0; v < V; ++v) y[v] = *reinterpret_cast<const float4*>(&Bs[tx + 16 * v][k]);
#pragma unroll
        for (int u = 0; u < U; ++u)
#pragma unroll
          for (int v = 0; v < V; ++v)
            acc[u][v] = fmaf(x[u].w, y[v].w, fmaf(x[u].z, y[v].z, fmaf(x[u].y, y[v].y, fmaf(x[u].x, y[v].x, acc[u][v]))));
      }
    }
    if (tid < M)
#pragma unroll
      for (int k = 0; k < DW_K; ++k) bsum += As[tid][k];
    __syncthreads();
  }
#pragma unroll
  for (int u = 0; u < U; ++u)
#pragma unroll
    for (int v = 0; v < V; ++v) {
      const int o = ty + 16 * u, c = tx + 16 * v;
      if (o < M && c < C) W[o * C + c] = acc[u][v];
    }
  if (tid < M) b[tid] = bsum;
}
__global__ void __launch_bounds__(256) k_ws_dw(const float* __restrict__ act, const float* __restrict__ del, long long np,
                                               long long chunk, float* __restrict__ partial) {
  __shared__ __align__(16) float As[64][DW_LD], Bs[64][DW_LD];
  float* P = partial + (size_t)blockIdx.x * WsTC::PARAMS;
  if (blockIdx.y == 0)
    ws_dw_layer<WsTC::H1, WsTC::K0>(As, Bs, del, act, np, chunk, P + WsTC::F_W1, P + WsTC::F_B1);
  else if (blockIdx.y == 1)
    ws_dw_layer<WsTC::H2, WsTC::H1>(As, Bs, del + (size_t)WsTC::H1 * np, act + (size_t)WsTC::K0 * np, np, chunk,
                                    P + WsTC::F_W2, P + WsTC::F_B2);
  else
    ws_dw_layer<WsTC::NO, WsTC::H2>(As, Bs, del + (size_t)(WsTC::H1 + WsTC::H2) * np,
                                    act + (size_t)(WsTC::K0 + WsTC::H1) * np, np, chunk, P + WsTC::F_W3, P + WsTC::F_B3);
}

// The splits' partials added up in a fixed order, 32 parameters a block, eight threads each; the last
// block sums the warps' squared errors (fixed strided order, then a tree).
__global__ void __launch_bounds__(256) k_ws_sum(const float* __restrict__ partial, int splits, float* __restrict__ dW,
                                                const float* __restrict__ loss_part, long long warps, float inv_n,
                                                float* __restrict__ loss) {
  __shared__ float red[256];
  const int tid = threadIdx.x;
  float s = 0.f;
  if (blockIdx.x + 1 == gridDim.x) {
    for (long long k = tid; k < warps; k += 256) s += loss_part[k];
    red[tid] = s;
    __syncthreads();
    for (int w = 128; w > 0; w >>= 1) {
      if (tid < w) red[tid] += red[tid + w];
      __syncthreads();
    }
    if (tid == 0) *loss = red[0] * inv_n;
    return;
  }
  const int p = blockIdx.x * 32 + (tid & 31), q0 = tid >> 5;
  if (p < WsTC::PARAMS)
#pragma unroll 4
    for (int q = q0; q < splits; q += 8) s += partial[(size_t)q * WsTC::PARAMS + p];
  red[tid] = s;
  __syncthreads();
  if (tid < 32 && p < WsTC::PARAMS) {
#pragma unroll
    for (int q = 1; q < 8; ++q) s += red[tid + 32 * q];
    dW[p] = s;
  }
}

// Adam (Kingma and Ba, 2015) on fp32 parameters with bias-corrected moments.
__global__ void k_adam(float* W, const float* __restrict__ g, float* m, float* v, long long count, float lr, float b1,
                       float b2, float eps, float c1, float c2) {
  const long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= count) return;
  const float gk = g[k];
  const float mk = b1 * m[k] + (1.f - b1) * gk;
  const float vk = b2 * v[k] + (1.f - b2) * gk * gk;
  m[k] = mk;
  v[k] = vk;
  W[k] -= lr * (mk / c1) / (sqrtf(vk / c2) + eps);
}

long long round32(long long n) { return (n + 31) / 32 * 32; }
int splits_for(long long np) { return (int)std::min<long long>(256, (np + 255) / 256); }

// Workspace carve-up (floats): tensor-core weights, biases, activations, deltas, split-K
// partials, per-warp loss partials.
struct WsWork {
  __nv_bfloat16* tc;
  float *bias, *act, *del, *partial, *loss_part;
};
WsWork carve(float* work, long long n) {
  const long long np = round32(n);
  WsWork w;
  float* p = work;
  w.tc = reinterpret_cast<__nv_bfloat16*>(p);
  p += (WsTC::SIZE + 1) / 2 + 64;
  w.bias = p;
  p += WsTC::BSIZE + 56;
  w.act = p;
  p += (size_t)ACT_ROWS * np;
  w.del = p;
  p += (size_t)DEL_ROWS * np;
  w.partial = p;
  p += (size_t)splits_for(np) * WsTC::PARAMS;
  w.loss_part = p;
  return w;
}

}  // namespace

cudaError_t launch_ws_prep(const float* W, __nv_bfloat16* tc, float* bias, cudaStream_t s) {
  k_ws_prep<<<(WsTC::SIZE + 255) / 256, 256, 0, s>>>(W, tc, bias);
  return cudaGetLastError();
}

extern "C" {

int64_t dp_ws_workspace_floats(int64_t n) {
  if (n < 0) return -1;
  const long long np = round32(std::max<long long>(n, 1));
  return (WsTC::SIZE + 1) / 2 + 64 + WsTC::BSIZE + 56 + (long long)(ACT_ROWS + DEL_ROWS) * np +
         (long long)splits_for(np) * WsTC::PARAMS + np / 32 + 32;
}

int32_t dp_ws_param_count(void) { return WsTC::PARAMS; }

dp_status dp_ws_forward(const float* W, const float* feats, int64_t n, float* y, float* work, void* stream) {
  if (!W || !feats || !y || !work || n < 0) return dp_internal_fail(DP_EINVAL, "dp_ws_forward: NULL pointer or n < 0");
  if (n == 0) return DP_OK;
  cudaStream_t s = (cudaStream_t)stream;
  WsWork w = carve(work, n);
  k_ws_prep<<<(WsTC::SIZE + 255) / 256, 256, 0, s>>>(W, w.tc, w.bias);
  const long long warps = round32(n) / 32;
  k_ws_infer<<<(unsigned)((warps + WS_WARPS - 1) / WS_WARPS), 32 * WS_WARPS, 0, s>>>(w.tc, w.bias, feats, WsTC::K0, n, y);
  cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? DP_OK : dp_internal_fail(DP_ECUDA, cudaGetErrorString(e));
}

dp_status dp_ws_loss_grad(const float* W, const float* rows, int64_t n, float* loss, float* dW, float* work,
                          void* stream) {
  if (!W || !rows || !loss || !dW || !work || n <= 0)
    return dp_internal_fail(DP_EINVAL, "dp_ws_loss_grad: NULL pointer or n <= 0");
  cudaStream_t s = (cudaStream_t)stream;
  const long long np = round32(n);
  WsWork w = carve(work, n);
  k_ws_prep<<<(WsTC::SIZE + 255) / 256, 256, 0, s>>>(W, w.tc, w.bias);
  const long long warps = np / 32;
  k_ws_fwdbwd<<<(unsigned)((warps + WS_WARPS - 1) / WS_WARPS), 32 * WS_WARPS, 0, s>>>(
      w.tc, w.bias, rows, n, np, 1.f / (float)n, w.act, w.del, w.loss_part);
  // dW_l = sum over rows of delta_l (x) act_l, db_l = sum of delta_l
  const int splits = splits_for(np);
  const long long chunk = ((np + splits - 1) / splits + DW_K - 1) / DW_K * DW_K;
  k_ws_dw<<<dim3(splits, 3), 256, 0, s>>>(w.act, w.del, np, chunk, w.partial);
  k_ws_sum<<<(WsTC::PARAMS + 31) / 32 + 1, 256, 0, s>>>(w.partial, splits, dW, w.loss_part, warps, 1.f / (float)n, loss);
  cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? DP_OK : dp_internal_fail(DP_ECUDA, cudaGetErrorString(e));
}

dp_status dp_ws_adam(float* W, const float* dW, float* m, float* v, int64_t count, int32_t step, float lr, float beta1,
                     float beta2, float eps, void* stream) {
  if (!W || !dW || !m || !v || count < 0 || step < 1)
    return dp_internal_fail(DP_EINVAL, "dp_ws_adam: NULL pointer, count < 0 or step < 1");
  if (count == 0) return DP_OK;
  const float c1 = 1.f - powf(beta1, (float)step), c2 = 1.f - powf(beta2, (float)step);
  k_adam<<<(unsigned)((count + 255) / 256), 256, 0, (cudaStream_t)stream>>>(W, dW, m, v, count, lr, beta1, beta2, eps,
                                                                            c1, c2);
  cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? DP_OK : dp_internal_fail(DP_ECUDA, cudaGetErrorString(e));
}

}  // extern "C"
