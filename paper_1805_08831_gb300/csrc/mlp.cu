// The learned scheduler's network: an FP32 multilayer perceptron 8 -> 32 -> 32 -> 2 with ReLU
// hidden layers, evaluated and trained by the kernels below (no library calls).
//
// Parameters (1410 floats, row-major, in this order): W1[8][32], b1[32], W2[32][32], b2[32],
// W3[32][2], b3[2]; W[i][j] connects input i to output j. Outputs: out[0] = predicted
// log2(1 + |C|) (cavity size), out[1] = logit of the probability that the point loses a
// conflict at least once. Loss of one sample with targets (y0, y1):
//   (out[0] - y0)^2 + softplus(out[1]) - y1 * out[1]      (squared error + binary cross-entropy)
// averaged over the samples.
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>

#include "internal.h"

namespace cg = cooperative_groups;

namespace dtg {
namespace {

constexpr int kIn = 8, kH = 32, kOut = 2;
constexpr int kOffW1 = 0, kOffB1 = kOffW1 + kIn * kH, kOffW2 = kOffB1 + kH, kOffB2 = kOffW2 + kH * kH,
              kOffW3 = kOffB2 + kH, kOffB3 = kOffW3 + kH * kOut, kParams = kOffB3 + kOut;
static_assert(kParams == 1410, "parameter count");
constexpr int kMlpThreads = 256;
constexpr float kBeta1 = 0.9f, kBeta2 = 0.999f, kAdamEps = 1e-8f;  // Adam

__device__ __forceinline__ float softplus(float z) { return z > 20.f ? z : log1pf(__expf(z)); }
__device__ __forceinline__ float sigmoid(float z) { return 1.f / (1.f + __expf(-z)); }

__device__ __forceinline__ uint64_t mix64(uint64_t z) {
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}

// Forward pass of one sample.
__device__ __forceinline__ void mlp_forward(const float* __restrict__ P, const float* x, float* h1, float* h2,
                                            float* out) {
  for (int j = 0; j < kH; ++j) {
    float a = P[kOffB1 + j];
    for (int i = 0; i < kIn; ++i) a = fmaf(x[i], P[kOffW1 + i * kH + j], a);
    h1[j] = fmaxf(a, 0.f);
  }
  for (int j = 0; j < kH; ++j) {
    float a = P[kOffB2 + j];
    for (int i = 0; i < kH; ++i) a = fmaf(h1[i], P[kOffW2 + i * kH + j], a);
    h2[j] = fmaxf(a, 0.f);
  }
  for (int j = 0; j < kOut; ++j) {
    float a = P[kOffB3 + j];
    for (int i = 0; i < kH; ++i) a = fmaf(h2[i], P[kOffW3 + i * kOut + j], a);
    out[j] = a;
  }
}

__global__ void __launch_bounds__(kMlpThreads) k_mlp_forward(const float* __restrict__ params,
                                                             const float* __restrict__ x, uint64_t n,
                                                             float* __restrict__ out) {
  __shared__ float P[kParams];
  for (int i = threadIdx.x; i < kParams; i += blockDim.x) P[i] = params[i];
  __syncthreads();
  for (uint64_t s = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; s < n; s += (uint64_t)gridDim.x * blockDim.x) {
    float xi[kIn], h1[kH], h2[kH], o[kOut];
    for (int i = 0; i < kIn; ++i) xi[i] = x[s * kIn + i];
    mlp_forward(P, xi, h1, h2, o);
    out[s * kOut] = o[0];
    out[s * kOut + 1] = o[1];
  }
}

// One step over n samples (rows 0 .. n, or with kDraw the minibatch drawn by a counter-based hash
// of draw_seed from `rows` rows): the mean loss and its gradient are added into loss[0] and
// grad[kParams], and with kDraw the last block to finish makes the Adam step and clears grad for
// the next one.
//
// A block takes tiles of 32 samples and runs the layers as small matrix products in shared
// memory, lane = hidden unit: forward, then backward, the products over the samples (the
// weights' gradients) accumulated in registers over all of a block's tiles. The eight blocks of a
// cluster then add up their parts through shared memory, so that a minibatch of 4096 adds 16
// terms to an entry in global memory, not 128: a longer chain rounds more (the loss of one step
// was off by 2.9e-7 instead of 0.6e-7; with a shared copy per block 0.7e-7). What bounds a training
// step is latency (one launch, one gather of random rows, the layers' chain, one round of
// atomics; 0.02 ms): a minibatch of 4096 takes 33 MFLOP. Adding every sample's 1410 products to
// one shared copy with atomics, as a thread per sample, serialised the lanes on one address each
// and took 1.3 ms a step.
constexpr int kS = 32;       // samples per tile
constexpr int kCluster = 8;  // blocks that add up their parts before they go to global memory

template <bool kDraw>
__global__ void __cluster_dims__(kCluster, 1, 1) __launch_bounds__(kMlpThreads) k_mlp_step(float* params, const float* __restrict__ x,
                                                          const float* __restrict__ y, uint64_t n, uint64_t rows,
                                                          uint64_t draw_seed, float scale, float* grad, float* loss,
                                                          unsigned int* ticket, float* m, float* v, float lr, int t) {
  __shared__ float W1[kIn][kH], W2[kH][kH + 1], W3[kH][kOut], B[kH + kH + kOut];
  __shared__ float X[kS][kIn], Y[kS][kOut], H1[kS][kH], H2[kS][kH], D1[kS][kH], D2[kS][kH], D3[kS][kOut];
  __shared__ uint64_t row[kS];
  __shared__ unsigned int s_last;
  constexpr int kWarps = kMlpThreads / 32;
  __shared__ float G[kParams + 1], s_sum[kWarps];
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  for (int i = tid; i < kIn * kH; i += kMlpThreads) W1[i / kH][i % kH] = __ldcg(&params[kOffW1 + i]);
  for (int i = tid; i < kH * kH; i += kMlpThreads) W2[i / kH][i % kH] = __ldcg(&params[kOffW2 + i]);
  for (int i = tid; i < kH * kOut; i += kMlpThreads) W3[i / kOut][i % kOut] = __ldcg(&params[kOffW3 + i]);
  for (int i = tid; i < kH; i += kMlpThreads) {
    B[i] = __ldcg(&params[kOffB1 + i]);
    B[kH + i] = __ldcg(&params[kOffB2 + i]);
  }
  if (tid < kOut) B[2 * kH + tid] = __ldcg(&params[kOffB3 + tid]);
  // this thread's entries of the gradient: W2[wid + kWarps k][lane], W1[wid][lane], and for the
  // first threads W3[tid / 2][tid % 2] and the biases
  float g2[kH / kWarps] = {}, g1 = 0.f, g3 = 0.f, gb1 = 0.f, gb2 = 0.f, gb3 = 0.f, sum = 0.f;
  static_assert(kWarps == kIn && kH == 32 && kOut == 2, "the tiling below");
  for (uint64_t s0 = (uint64_t)blockIdx.x * kS; s0 < n; s0 += (uint64_t)gridDim.x * kS) {
    const int ns = (int)min((unsigned long long)kS, (unsigned long long)(n - s0));
    __syncthreads();  // the parameters are in place; the last tile's products are done
    if (tid < kS) {
      const uint64_t k = s0 + tid;
      row[tid] = kDraw ? mix64(draw_seed + 0x9E3779B97F4A7C15ull * (k + 1)) % rows : k;
    }
    __syncthreads();
    {
      const int s = tid / kIn, i = tid % kIn;
      X[s][i] = s < ns ? x[row[s] * kIn + i] : 0.f;
      if (tid < kS * kOut) Y[tid / kOut][tid % kOut] = tid / kOut < ns ? y[row[tid / kOut] * kOut + tid % kOut] : 0.f;
    }
    __syncthreads();
    // a warp's four samples go through a layer together: four independent sums per weight read
    constexpr int kPer = kS / kWarps;
    float h[kPer];
#pragma unroll
    for (int q = 0; q < kPer; ++q) {
      float a = B[lane];
      for (int i = 0; i < kIn; ++i) a = fmaf(X[wid + kWarps * q][i], W1[i][lane], a);
      H1[wid + kWarps * q][lane] = fmaxf(a, 0.f);
    }
    __syncwarp();  // a sample stays with its warp until the products over the samples
#pragma unroll
    for (int q = 0; q < kPer; ++q) h[q] = B[kH + lane];
#pragma unroll 8
    for (int i = 0; i < kH; ++i) {
      const float wt = W2[i][lane];
#pragma unroll
      for (int q = 0; q < kPer; ++q) h[q] = fmaf(H1[wid + kWarps * q][i], wt, h[q]);
    }
#pragma unroll
    for (int q = 0; q < kPer; ++q) {
      const int s = wid + kWarps * q;
      h[q] = fmaxf(h[q], 0.f);
      H2[s][lane] = h[q];
      float o0 = h[q] * W3[lane][0], o1 = h[q] * W3[lane][1];
      for (int d = 16; d > 0; d >>= 1) {
        o0 += __shfl_xor_sync(0xFFFFFFFFu, o0, d);
        o1 += __shfl_xor_sync(0xFFFFFFFFu, o1, d);
      }
      o0 += B[2 * kH];
      o1 += B[2 * kH + 1];
      const float y0 = Y[s][0], y1 = Y[s][1], e = o0 - y0;
      if (lane == 0 && s < ns) sum += scale * (e * e + softplus(o1) - y1 * o1);
      const float d0 = s < ns ? 2.f * e * scale : 0.f, d1 = s < ns ? (sigmoid(o1) - y1) * scale : 0.f;
      if (lane < kOut) D3[s][lane] = lane == 0 ? d0 : d1;
      D2[s][lane] = h[q] > 0.f ? d0 * W3[lane][0] + d1 * W3[lane][1] : 0.f;
    }
    __syncwarp();
#pragma unroll
    for (int q = 0; q < kPer; ++q) h[q] = 0.f;
#pragma unroll 8
    for (int j = 0; j < kH; ++j) {
      const float wt = W2[lane][j];
#pragma unroll
      for (int q = 0; q < kPer; ++q) h[q] = fmaf(D2[wid + kWarps * q][j], wt, h[q]);
    }
#pragma unroll
    for (int q = 0; q < kPer; ++q)
      D1[wid + kWarps * q][lane] = H1[wid + kWarps * q][lane] > 0.f ? h[q] : 0.f;
    __syncthreads();
#pragma unroll 4
    for (int s = 0; s < kS; ++s) {  // a unit without a gradient takes no part, whatever its input
      const float d2 = D2[s][lane], d1 = D1[s][lane];
      for (int k = 0; k < kH / kWarps; ++k) g2[k] = d2 != 0.f ? fmaf(H1[s][wid + kWarps * k], d2, g2[k]) : g2[k];
      g1 = d1 != 0.f ? fmaf(X[s][wid], d1, g1) : g1;
    }
    if (tid < kH * kOut)
      for (int s = 0; s < kS; ++s) g3 = fmaf(H2[s][tid / kOut], D3[s][tid % kOut], g3);
    else if (tid < kH * kOut + kH)
      for (int s = 0; s < kS; ++s) gb1 += D1[s][lane];
    else if (tid < kH * kOut + 2 * kH)
      for (int s = 0; s < kS; ++s) gb2 += D2[s][lane];
    else if (tid < kH * kOut + 2 * kH + kOut)
      for (int s = 0; s < kS; ++s) gb3 += D3[s][lane];
  }
  // the cluster's blocks add up their parts, an eighth of the entries each
  for (int k = 0; k < kH / kWarps; ++k) G[kOffW2 + (wid + kWarps * k) * kH + lane] = g2[k];
  G[kOffW1 + wid * kH + lane] = g1;
  if (tid < kH * kOut) G[kOffW3 + tid] = g3;
  else if (tid < kH * kOut + kH) G[kOffB1 + lane] = gb1;
  else if (tid < kH * kOut + 2 * kH) G[kOffB2 + lane] = gb2;
  else if (tid < kH * kOut + 2 * kH + kOut) G[kOffB3 + lane] = gb3;
  if (lane == 0) s_sum[wid] = sum;
  __syncthreads();
  if (tid == 0) {
    float l = 0.f;
    for (int k = 0; k < kWarps; ++k) l += s_sum[k];
    G[kParams] = l;
  }
  cg::cluster_group cluster = cg::this_cluster();
  cluster.sync();
  for (int i = (int)cluster.block_rank() + kCluster * tid; i <= kParams; i += kCluster * kMlpThreads) {
    float part[kCluster], a = 0.f;
    for (int r = 0; r < kCluster; ++r) part[r] = cluster.map_shared_rank(G, r)[i];
    for (int r = 0; r < kCluster; ++r) a += part[r];
    atomicAdd(i < kParams ? &grad[i] : loss, a);
  }
  if constexpr (kDraw) __threadfence();
  cluster.sync();  // every block's part has been read, and this block's sums are on their way
  if constexpr (kDraw) {
    // the last block to add its part holds the whole gradient
    if (tid == 0) s_last = atomicAdd(ticket, 1u) == gridDim.x - 1 ? 1u : 0u;
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    if (tid == 0) *ticket = 0;
    const float c1 = 1.f - powf(kBeta1, (float)t), c2 = 1.f - powf(kBeta2, (float)t);
    for (int i = tid; i < kParams; i += kMlpThreads) {
      const float g = __ldcg(&grad[i]);
      const float mi = kBeta1 * m[i] + (1.f - kBeta1) * g;
      const float vi = kBeta2 * v[i] + (1.f - kBeta2) * g * g;
      m[i] = mi;
      v[i] = vi;
      params[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + kAdamEps);
      grad[i] = 0.f;
    }
  }
}

// Blocks of a step: one tile each while that fills the chip, then tiles are taken in turn; whole
// clusters.
unsigned step_grid(uint64_t n) {
  const uint64_t b = std::max<uint64_t>(1, std::min<uint64_t>((n + kS - 1) / kS, 152ull * 4));
  return (unsigned)((b + kCluster - 1) / kCluster * kCluster);
}

unsigned mlp_grid(uint64_t n) {
  uint64_t b = (n + kMlpThreads - 1) / kMlpThreads;
  return (unsigned)std::max<uint64_t>(1, std::min<uint64_t>(b, 152ull * 4));
}

}  // namespace

int mlp_params() { return kParams; }

int mlp_forward(const float* params, const float* x, uint64_t n, float* out, cudaStream_t s) {
  if (n == 0) return DT_OK;
  k_mlp_forward<<<mlp_grid(n), kMlpThreads, 0, s>>>(params, x, n, out);
  ++g_kernel_launches;
  return cudaPeekAtLastError() == cudaSuccess ? DT_OK : DT_ECUDA;
}

int mlp_grad(const float* params, const float* x, const float* y, uint64_t n, float* grad, float* loss,
             cudaStream_t s) {
  if (n == 0) return DT_EINVAL;
  cudaMemsetAsync(grad, 0, kParams * sizeof(float), s);
  cudaMemsetAsync(loss, 0, sizeof(float), s);
  k_mlp_step<false><<<step_grid(n), kMlpThreads, 0, s>>>(const_cast<float*>(params), x, y, n, n, 0, 1.f / (float)n,
                                                         grad, loss, nullptr, nullptr, nullptr, 0.f, 0);
  ++g_kernel_launches;
  return cudaPeekAtLastError() == cudaSuccess ? DT_OK : DT_ECUDA;
}

int mlp_train(float* params, const float* x, const float* y, uint64_t n, uint32_t steps, uint32_t batch, float lr,
              uint64_t seed, float* losses_host, cudaStream_t s) {
  if (n == 0 || batch == 0) return DT_EINVAL;
  // gradient, both moments, the ticket and the losses in one allocation
  float* ws = nullptr;
  const size_t entries = 3 * (size_t)kParams + 1 + std::max(steps, 1u);
  if (cudaMalloc(&ws, entries * 4) != cudaSuccess) return DT_ENOMEM;
  float *grad = ws, *m = grad + kParams, *v = m + kParams, *loss = v + kParams + 1;
  unsigned int* ticket = reinterpret_cast<unsigned int*>(v + kParams);
  cudaMemsetAsync(ws, 0, entries * 4, s);
  for (uint32_t t = 0; t < steps; ++t)
    k_mlp_step<true><<<step_grid(batch), kMlpThreads, 0, s>>>(params, x, y, batch, n, seed + 0x51ED2701ull * (t + 1),
                                                              1.f / (float)batch, grad, loss + t, ticket, m, v, lr,
                                                              (int)t + 1);
  g_kernel_launches += steps;
  int rc = cudaPeekAtLastError() == cudaSuccess ? DT_OK : DT_ECUDA;
  if (losses_host && steps && cudaMemcpyAsync(losses_host, loss, steps * 4ull, cudaMemcpyDeviceToHost, s) != cudaSuccess)
    rc = DT_ECUDA;
  if (cudaStreamSynchronize(s) != cudaSuccess) rc = DT_ECUDA;
  cudaFree(ws);
  return rc;
}

}  // namespace dtg
