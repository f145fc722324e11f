// Training and evaluation kernels of the learned Newton guess (FP32).
//
// Network: 6 -> 64 -> 64 -> 1, tanh hidden layers, linear output; loss: mean
// squared error over a batch; optimiser: Adam.  Parameter layout (4673):
// W1[6][64], b1[64], W2[64][64], b2[64], w3[64], b3.
// Per batch of n samples the caller provides a work array of
// GRP_MLP_WORK_FLOATS(n) floats: the blocks' partial gradients and losses.
#include <cuda_runtime.h>

#include "grp_device.cuh"
#include "grprec.h"

using grp::MLP_NH;
using grp::MLP_NIN;
using grp::MLP_NPARAM;

namespace {

constexpr int OFF_W1 = 0;
constexpr int OFF_B1 = OFF_W1 + MLP_NIN * MLP_NH;
constexpr int OFF_W2 = OFF_B1 + MLP_NH;
constexpr int OFF_B2 = OFF_W2 + MLP_NH * MLP_NH;
constexpr int OFF_W3 = OFF_B2 + MLP_NH;
constexpr int OFF_B3 = OFF_W3 + MLP_NH;

// A block takes tiles of 32 samples through the whole network with the weights
// and the tile's activations in shared memory: forward, and for training the
// loss, the back-propagation and the tile's share of every weight gradient,
// which the threads keep in registers over the block's tiles.  Each block then
// leaves one partial gradient, and k_mlp_reduce adds the partials.
//   256 threads: unit u = tid & 63 of a layer, samples 8 (tid / 64) ..+7 for the
//   two layers and their back-propagation; a 4 x 4 patch of W2's gradient.
//   W2's rows are 65 words apart (read along rows and along columns), the
//   tile's 68 (float4 reads).
// Bound by FP32 issue and, at a mini-batch of 4096 (128 blocks), by the latency
// of one tile.  The activations used to go through device memory, and 73 blocks
// summed the weight gradients sample by sample: 514 us for a training step of
// 4096 samples.
constexpr int TILE = 32, PITCH = 68, W2P = MLP_NH + 1;
constexpr int PARTIAL = MLP_NPARAM + 1;             // gradient and loss

struct MlpShared {
  float W1[MLP_NIN * MLP_NH], b1[MLP_NH], b2[MLP_NH], w3[MLP_NH];
  float W2[MLP_NH * W2P];
  float A[TILE * PITCH];                            // h1, then dz1
  float B[TILE * PITCH];                            // h2, then dz2
  float X[TILE * MLP_NIN], dy[TILE], red[256];
};

template <bool GRAD>
__global__ void __launch_bounds__(256) k_mlp_tiles(const float* __restrict__ w, const float* __restrict__ x,
                                                   const float* __restrict__ t, long long n, float* __restrict__ out,
                                                   float* __restrict__ loss_out)
{
  __shared__ __align__(16) MlpShared S;
  const int tid = threadIdx.x, u = tid & 63, s0 = (tid >> 6) * 8, warp = tid >> 5, lane = tid & 31;
  for (int i = tid; i < MLP_NIN * MLP_NH; i += 256) S.W1[i] = w[OFF_W1 + i];
  for (int i = tid; i < MLP_NH * MLP_NH; i += 256) S.W2[(i >> 6) * W2P + (i & 63)] = w[OFF_W2 + i];
  if (tid < MLP_NH) { S.b1[tid] = w[OFF_B1 + tid]; S.b2[tid] = w[OFF_B2 + tid]; S.w3[tid] = w[OFF_W3 + tid]; }
  const float b3 = w[OFF_B3];
  const int j4 = (tid >> 4) * 4, k4 = (tid & 15) * 4;
  float gW2[4][4], gW1[2] = {0.0f, 0.0f}, gw3 = 0.0f, gb1 = 0.0f, gb2 = 0.0f, gb3 = 0.0f, loss = 0.0f;
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int k = 0; k < 4; ++k) gW2[i][k] = 0.0f;
  const long long tiles = (n + TILE - 1) / TILE;
  for (long long tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
    const long long base = tile * TILE;
    __syncthreads();                                // the weights are there; the last tile is done with
    // (places past the end repeat the last sample with no weight: zeros would meet
    // an infinite weight as 0 x infinity)
    if (tid < TILE * MLP_NIN) {
      const long long s = base + tid / MLP_NIN;
      S.X[tid] = x[(s < n ? s : n - 1) * MLP_NIN + tid % MLP_NIN];
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      float z = S.b1[u];
#pragma unroll
      for (int i = 0; i < MLP_NIN; ++i) z = fmaf(S.X[(s0 + q) * MLP_NIN + i], S.W1[i * MLP_NH + u], z);
      S.A[(s0 + q) * PITCH + u] = tanhf(z);
    }
    __syncthreads();
    float z[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) z[q] = S.b2[u];
#pragma unroll 4
    for (int j = 0; j < MLP_NH; j += 4) {
      const float w0 = S.W2[j * W2P + u], w1 = S.W2[(j + 1) * W2P + u], w2 = S.W2[(j + 2) * W2P + u],
                  w3 = S.W2[(j + 3) * W2P + u];
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        const float4 h = *reinterpret_cast<const float4*>(&S.A[(s0 + q) * PITCH + j]);
        z[q] = fmaf(h.w, w3, fmaf(h.z, w2, fmaf(h.y, w1, fmaf(h.x, w0, z[q]))));
      }
    }
#pragma unroll
    for (int q = 0; q < 8; ++q) { z[q] = tanhf(z[q]); S.B[(s0 + q) * PITCH + u] = z[q]; }
    __syncthreads();
    // outputs: four samples per warp
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int sm = warp * 4 + q;
      float y = fmaf(S.B[sm * PITCH + lane], S.w3[lane], S.B[sm * PITCH + lane + 32] * S.w3[lane + 32]);
#pragma unroll
      for (int off = 16; off > 0; off >>= 1) y += __shfl_xor_sync(0xffffffffu, y, off);
      y += b3;
      if (lane == 0 && base + sm < n) {
        if (!GRAD) out[base + sm] = y;
        else {
          const float r = y - t[base + sm];
          loss = fmaf(r, r, loss);
          S.dy[sm] = 2.0f * r / (float)n;
        }
      } else if (GRAD && lane == 0) {
        S.dy[sm] = 0.0f;
      }
    }
    if (!GRAD) continue;
    __syncthreads();
    // dz2 in place of h2
    const float v3 = S.w3[u];
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const float dy = S.dy[s0 + q];
      gw3 = fmaf(z[q], dy, gw3);
      if (u == 0) gb3 += dy;
      const float dz = dy * v3 * (1.0f - z[q] * z[q]);
      gb2 += dz;
      S.B[(s0 + q) * PITCH + u] = dz;
    }
    __syncthreads();
#pragma unroll 4
    for (int sm = 0; sm < TILE; ++sm) {
      const float4 h = *reinterpret_cast<const float4*>(&S.A[sm * PITCH + j4]);
      const float4 d = *reinterpret_cast<const float4*>(&S.B[sm * PITCH + k4]);
      const float hh[4] = {h.x, h.y, h.z, h.w}, dd[4] = {d.x, d.y, d.z, d.w};
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int k = 0; k < 4; ++k) gW2[i][k] = fmaf(hh[i], dd[k], gW2[i][k]);
    }
    // dz1 = (dz2 W2^T) (1 - h1^2)
#pragma unroll
    for (int q = 0; q < 8; ++q) z[q] = 0.0f;
#pragma unroll 4
    for (int k = 0; k < MLP_NH; k += 4) {
      const float w0 = S.W2[u * W2P + k], w1 = S.W2[u * W2P + k + 1], w2 = S.W2[u * W2P + k + 2],
                  w3 = S.W2[u * W2P + k + 3];
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        const float4 d = *reinterpret_cast<const float4*>(&S.B[(s0 + q) * PITCH + k]);
        z[q] = fmaf(d.w, w3, fmaf(d.z, w2, fmaf(d.y, w1, fmaf(d.x, w0, z[q]))));
      }
    }
    __syncthreads();                                // every read of h1 as a factor is done
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const float h = S.A[(s0 + q) * PITCH + u], dz = z[q] * (1.0f - h * h);
      gb1 += dz;
      S.A[(s0 + q) * PITCH + u] = dz;
    }
    __syncthreads();
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      const int o = tid + 256 * e;
      if (o < MLP_NIN * MLP_NH) {
#pragma unroll 8
        for (int sm = 0; sm < TILE; ++sm) gW1[e] = fmaf(S.X[sm * MLP_NIN + (o >> 6)], S.A[sm * PITCH + (o & 63)], gW1[e]);
      }
    }
  }
  if (!GRAD) return;
  float* g = out + (long long)blockIdx.x * PARTIAL;
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int k = 0; k < 4; ++k) g[OFF_W2 + (j4 + i) * MLP_NH + k4 + k] = gW2[i][k];
  g[OFF_W1 + tid] = gW1[0];
  if (tid + 256 < MLP_NIN * MLP_NH) g[OFF_W1 + 256 + tid] = gW1[1];
  // the vectors: four partial sums (sample groups) per unit
  const float part[3] = {gb1, gb2, gw3};
  const int dst[3] = {OFF_B1, OFF_B2, OFF_W3};
#pragma unroll
  for (int e = 0; e < 3; ++e) {
    __syncthreads();
    S.red[tid] = part[e];
    __syncthreads();
    if (tid < 64) g[dst[e] + u] = (S.red[u] + S.red[64 + u]) + (S.red[128 + u] + S.red[192 + u]);
  }
  __syncthreads();
  S.red[tid] = lane == 0 ? loss : 0.0f;
  if (u == 0) S.dy[tid >> 6] = gb3;
  __syncthreads();
  if (tid == 0) {
    float l = 0.0f;
    for (int k = 0; k < 8; ++k) l += S.red[32 * k];
    if (loss_out) *loss_out = l / (float)n;          // the only block: its partial is the gradient
    else g[MLP_NPARAM] = l;
    g[OFF_B3] = (S.dy[0] + S.dy[1]) + (S.dy[2] + S.dy[3]);
  }
}

// Sum of the blocks' partials: 32 outputs per block, eight threads each.
__global__ void __launch_bounds__(256) k_mlp_reduce(const float* __restrict__ part, int blocks, long long n,
                                                    float* __restrict__ grad, float* __restrict__ loss)
{
  __shared__ float red[8][33];
  const int o = blockIdx.x * 32 + (threadIdx.x & 31), slice = threadIdx.x >> 5;
  float s = 0.0f;
  if (o < PARTIAL) {
#pragma unroll 8
    for (int b = slice; b < blocks; b += 8) s += part[(long long)b * PARTIAL + o];
  }
  red[slice][threadIdx.x & 31] = s;
  __syncthreads();
  if (slice == 0 && o < PARTIAL) {
    float v = 0.0f;
#pragma unroll
    for (int k = 0; k < 8; ++k) v += red[k][threadIdx.x];
    if (o < MLP_NPARAM) grad[o] = v;
    else *loss = v / (float)n;
  }
}

__global__ void k_mlp_adam(float* __restrict__ w, const float* __restrict__ g, float* __restrict__ m,
                           float* __restrict__ v, int n, float lr, float beta1, float beta2, float eps,
                           float c1, float c2)
{
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const float gi = g[i];
  const float mi = beta1 * m[i] + (1.0f - beta1) * gi;
  const float vi = beta2 * v[i] + (1.0f - beta2) * gi * gi;
  m[i] = mi;
  v[i] = vi;
  w[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
}

}  // namespace

extern "C" {

int grp_mlp_forward(const float* weights, const float* x, long long n, float* y, void* stream)
{
  if (!weights || !x || !y || n < 0) return GRP_E_INVALID_ARG;
  if (n == 0) return GRP_OK;
  const long long tiles = (n + TILE - 1) / TILE;
  const unsigned g = (unsigned)(tiles < 608 ? tiles : 608);
  k_mlp_tiles<false><<<g, 256, 0, (cudaStream_t)stream>>>(weights, x, nullptr, n, y, nullptr);
  return cudaGetLastError() == cudaSuccess ? GRP_OK : GRP_E_CUDA;
}

int grp_mlp_loss_grad(const float* weights, const float* x, const float* target, long long n, float* grad,
                      float* loss, float* work, void* stream)
{
  if (!weights || !x || !target || !grad || !loss || !work || n < 1) return GRP_E_INVALID_ARG;
  cudaStream_t s = (cudaStream_t)stream;
  // one partial gradient per block, as many blocks as the scratch holds and two
  // per SM, the tiles spread evenly
  const long long tiles = (n + TILE - 1) / TILE;
  long long nb = GRP_MLP_WORK_FLOATS(n) / PARTIAL;
  nb = nb < 304 ? nb : 304;
  nb = nb < 1 ? 1 : nb;
  const long long each = (tiles + nb - 1) / nb;
  nb = (tiles + each - 1) / each;
  if (nb == 1) {
    k_mlp_tiles<true><<<1, 256, 0, s>>>(weights, x, target, n, grad, loss);
  } else {
    k_mlp_tiles<true><<<(unsigned)nb, 256, 0, s>>>(weights, x, target, n, work, nullptr);
    k_mlp_reduce<<<(PARTIAL + 31) / 32, 256, 0, s>>>(work, (int)nb, n, grad, loss);
  }
  return cudaGetLastError() == cudaSuccess ? GRP_OK : GRP_E_CUDA;
}

int grp_mlp_adam(float* weights, const float* grad, float* m, float* v, int step, float lr, float beta1,
                 float beta2, float eps, void* stream)
{
  if (!weights || !grad || !m || !v || step < 1) return GRP_E_INVALID_ARG;
  const float c1 = 1.0f - powf(beta1, (float)step), c2 = 1.0f - powf(beta2, (float)step);
  k_mlp_adam<<<(MLP_NPARAM + 255) / 256, 256, 0, (cudaStream_t)stream>>>(weights, grad, m, v, MLP_NPARAM, lr,
                                                                          beta1, beta2, eps, c1, c2);
  return cudaGetLastError() == cudaSuccess ? GRP_OK : GRP_E_CUDA;
}

}  // extern "C"
