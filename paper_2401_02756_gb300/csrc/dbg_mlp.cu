// K8: the capacity predictor's network -- FP32, 1024 -> 64 -> 64 -> 1 with
// ReLU, mapping a sketch's registers (scaled to [0, 1]) to ln(distinct
// vertices).  Forward, backward (mean squared error) and an Adam step, all
// in this file's kernels; no library calls.
//
// The arithmetic is small (100 MFLOP a training step of 256 rows, about 2 us
// of FP32 throughput; tensor cores would round the operands), so the time is
// launches and dependent latency.  A forward pass is one kernel and a training
// step two: everything of a row -- its forward pass, its loss derivative and
// the gradients of its hidden units -- is done by one CTA, then every
// parameter's gradient and Adam update by the CTA that sums it.  Step of 256
// rows: 165 us of kernels in 15 launches (GEMMs of 16 CTAs over a serial K of
// 1024, one-CTA column sums) -> 23 us a step, launches included (176 before).
//
// Parameter layout (DBG_MLP_PARAMS floats): W1 [64][1024] | b1 [64] |
// W2 [64][64] | b2 [64] | w3 [64] | b3 [1].
#include <math.h>

#include "dbg_internal.cuh"

namespace dbg {
namespace {

constexpr int kIn = DBG_MLP_INPUTS, kHid = DBG_MLP_HIDDEN;
constexpr int kOffW1 = 0, kOffB1 = kOffW1 + kHid * kIn, kOffW2 = kOffB1 + kHid,
              kOffB2 = kOffW2 + kHid * kHid, kOffW3 = kOffB2 + kHid, kOffB3 = kOffW3 + kHid;
static_assert(kOffB3 + 1 == DBG_MLP_PARAMS, "parameter layout");

struct Work {
  float *h1, *h2, *y, *dh1, *dh2, *dy, *loss;
};

constexpr int kRows = 2;     // rows of the batch per CTA: 256 rows fill 128 SMs
constexpr int kWarps = 8;    // warps per CTA

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int d = 16; d > 0; d >>= 1) v += __shfl_xor_sync(0xffffffffu, v, d);
  return v;
}

// kRows rows of the batch: y = the network's output; TRAIN: also dy = (y - t)
// / B and the gradients with respect to the hidden units before their ReLU,
// with the hidden units themselves, into `w`.  A warp takes a hidden unit at a
// time, its lanes the inputs (weights read coalesced, the rows' inputs held in
// registers), and sums over the lanes.
template <bool TRAIN>
__global__ void __launch_bounds__(32 * kWarps)
    k_rows(const float *P, const float *x, const float *target, int B, float *y, Work w) {
  after_previous();
  __shared__ float s_h1[kRows][kHid], s_h2[kRows][kHid], s_dh2[kRows][kHid];
  __shared__ float s_part[kRows][kHid], s_dy[kRows];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t r0 = (int64_t)blockIdx.x * kRows;
  constexpr int C = kIn / 32;
  float xr[kRows][C];
#pragma unroll
  for (int r = 0; r < kRows; ++r)
#pragma unroll
    for (int c = 0; c < C; ++c)
      xr[r][c] = r0 + r < B ? x[(r0 + r) * kIn + c * 32 + lane] : 0.f;
  // H1 = relu(X W1^T + b1)
#pragma unroll 2
  for (int j = warp; j < kHid; j += kWarps) {
    const float *row = P + kOffW1 + j * kIn + lane;
    float a[kRows] = {};
#pragma unroll
    for (int c = 0; c < C; ++c) {
      const float v = row[c * 32];
#pragma unroll
      for (int r = 0; r < kRows; ++r) a[r] += xr[r][c] * v;
    }
#pragma unroll
    for (int r = 0; r < kRows; ++r) {
      const float sum = warp_sum(a[r]);
      if (lane == r) s_h1[r][j] = fmaxf(sum + P[kOffB1 + j], 0.f);
    }
  }
  __syncthreads();
  // H2 = relu(H1 W2^T + b2)
#pragma unroll 4
  for (int j = warp; j < kHid; j += kWarps) {
    const float v0 = P[kOffW2 + j * kHid + lane], v1 = P[kOffW2 + j * kHid + 32 + lane];
#pragma unroll
    for (int r = 0; r < kRows; ++r) {
      const float sum = warp_sum(s_h1[r][lane] * v0 + s_h1[r][32 + lane] * v1);
      if (lane == r) s_h2[r][j] = fmaxf(sum + P[kOffB2 + j], 0.f);
    }
  }
  __syncthreads();
  // y = H2 w3 + b3
  if (warp < kRows) {
    const int r = warp;
    const float out = warp_sum(s_h2[r][lane] * P[kOffW3 + lane] +
                               s_h2[r][32 + lane] * P[kOffW3 + 32 + lane]) +
                      P[kOffB3];
    if (lane == 0 && r0 + r < B) {
      y[r0 + r] = out;
      if (TRAIN) {
        const float dy = (out - target[r0 + r]) / (float)B;
        s_dy[r] = dy;
        w.dy[r0 + r] = dy;
      }
    }
  }
  if constexpr (TRAIN) {
    __syncthreads();
    // dH2 = (dy w3) * relu'(H2), dH1 = (dH2 W2) * relu'(H1): a thread per
    // (row, hidden unit) and half of the sum
    static_assert(2 * kRows * kHid == 32 * kWarps, "two threads per row and hidden unit");
    const int k = threadIdx.x & (kHid - 1), r = (threadIdx.x >> 6) & (kRows - 1);
    const int half = threadIdx.x >> 7;
    const bool in = r0 + r < B;
    const int64_t at = (r0 + r) * kHid + k;
    if (half == 0) {
      const float h2 = s_h2[r][k];
      const float g = in && h2 > 0.f ? s_dy[r] * P[kOffW3 + k] : 0.f;
      s_dh2[r][k] = g;
      if (in) {
        w.h1[at] = s_h1[r][k];
        w.h2[at] = h2;
        w.dh2[at] = g;
      }
    }
    __syncthreads();
    float g = 0.f;
#pragma unroll 16
    for (int j = 32 * half; j < 32 * half + 32; ++j) g += s_dh2[r][j] * P[kOffW2 + j * kHid + k];
    if (half) s_part[r][k] = g;
    __syncthreads();
    if (!half && in) w.dh1[at] = s_h1[r][k] > 0.f ? g + s_part[r][k] : 0.f;
  }
}

// Adam (Kingma & Ba 2015) with bias correction.
struct Adam {
  float *p, *g, *m, *v;
  float lr, b1, b2, eps, c1, c2;
  __device__ __forceinline__ void step(int i, float gi) const {
    const float mi = b1 * m[i] + (1.f - b1) * gi;
    const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
    g[i] = gi;
    m[i] = mi;
    v[i] = vi;
    p[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
  }
};

constexpr int kCols = 8;                        // columns of a weight matrix per CTA
constexpr int kGradW1 = kIn / kCols;            // CTAs of dW1, then
constexpr int kGradW2 = kHid / kCols;           // of dW2, then one for dw3, db3 and the loss
constexpr int kGradCtas = kGradW1 + kGradW2 + 1;
constexpr int kGradRows = 256;                  // rows staged at a time

// Every gradient and its Adam update, and the loss: dW1 = dH1^T X and dW2 =
// dH2^T H1 by kCols columns of all 64 rows per CTA (137 CTAs: one wave), a
// quarter of the batch per group of 64 threads; the first CTA of a layer sums
// its biases too.
__global__ void __launch_bounds__(256, 2)
    k_grads(const float *x, const float *target, int B, Work w, Adam ad) {
  after_previous();
  __shared__ __align__(16) float s_x[kGradRows][kCols];
  __shared__ float s_red[4][kHid][kCols + 1];
  const int j = threadIdx.x & (kHid - 1), group = threadIdx.x >> 6;
  if (blockIdx.x == kGradW1 + kGradW2) {
    // dw3 = H2^T dy; db3 = sum dy; loss = mean of (y - t)^2 / 2
    float a = 0.f, b = 0.f, l = 0.f;
#pragma unroll 8
    for (int r = group; r < B; r += 4) a += w.h2[(int64_t)r * kHid + j] * w.dy[r];
    for (int r = threadIdx.x; r < B; r += 256) {
      const float d = w.y[r] - target[r];
      b += w.dy[r];
      l += 0.5f * d * d / (float)B;
    }
    b = warp_sum(b);
    l = warp_sum(l);
    s_red[group][j][0] = a;
    if ((threadIdx.x & 31) == 0) {
      s_x[threadIdx.x >> 5][0] = b;
      s_x[threadIdx.x >> 5][1] = l;
    }
    __syncthreads();
    if (group == 0)
      ad.step(kOffW3 + j, (s_red[0][j][0] + s_red[1][j][0]) + (s_red[2][j][0] + s_red[3][j][0]));
    if (threadIdx.x == 64) {
      float sum[2] = {0.f, 0.f};
      for (int q = 0; q < 8; ++q) {
        sum[0] += s_x[q][0];
        sum[1] += s_x[q][1];
      }
      ad.step(kOffB3, sum[0]);
      *w.loss = sum[1];
    }
    return;
  }
  const bool first = blockIdx.x < kGradW1;  // layer 1 or 2
  const int i0 = kCols * (first ? (int)blockIdx.x : (int)blockIdx.x - kGradW1);
  const float *dh = first ? w.dh1 : w.dh2, *in = first ? x : w.h1;
  const int ld = first ? kIn : kHid;
  float acc[kCols] = {}, bias = 0.f;
  for (int b0 = 0; b0 < B; b0 += kGradRows) {
    const int rows = min(kGradRows, B - b0);
    for (int e = threadIdx.x; e < rows * kCols; e += 256)
      s_x[e / kCols][e % kCols] = in[(int64_t)(b0 + e / kCols) * ld + i0 + e % kCols];
    __syncthreads();
#pragma unroll 8
    for (int r = group; r < rows; r += 4) {
      const float d = dh[(int64_t)(b0 + r) * kHid + j];
      const float4 lo = *reinterpret_cast<const float4 *>(&s_x[r][0]);
      const float4 hi = *reinterpret_cast<const float4 *>(&s_x[r][4]);
      acc[0] += d * lo.x;
      acc[1] += d * lo.y;
      acc[2] += d * lo.z;
      acc[3] += d * lo.w;
      acc[4] += d * hi.x;
      acc[5] += d * hi.y;
      acc[6] += d * hi.z;
      acc[7] += d * hi.w;
      bias += d;
    }
    __syncthreads();
  }
#pragma unroll
  for (int q = 0; q < kCols; ++q) s_red[group][j][q] = acc[q];
  s_red[group][j][kCols] = bias;
  __syncthreads();
  auto total = [&](int jj, int q) {
    return (s_red[0][jj][q] + s_red[1][jj][q]) + (s_red[2][jj][q] + s_red[3][jj][q]);
  };
  for (int e = threadIdx.x; e < kHid * kCols; e += 256) {
    const int jj = e / kCols, q = e % kCols;
    ad.step((first ? kOffW1 : kOffW2) + jj * ld + i0 + q, total(jj, q));
  }
  if (i0 == 0 && threadIdx.x < kHid) ad.step((first ? kOffB1 : kOffB2) + j, total(j, kCols));
}

// He-uniform initial weights from a counter-based hash (SplitMix64 of the
// parameter index), biases zero.
__global__ void k_init(float *p, uint64_t seed) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < DBG_MLP_PARAMS;
       i += gridDim.x * blockDim.x) {
    uint64_t z = seed + (uint64_t)(i + 1) * 0x9E3779B97F4A7C15ull;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    z ^= z >> 31;
    const float u = (float)(z >> 40) * (1.0f / 16777216.0f) * 2.f - 1.f;  // [-1, 1)
    float v = 0.f;
    if (i < kOffB1) v = u * sqrtf(6.f / kIn);
    else if (i >= kOffW2 && i < kOffB2) v = u * sqrtf(6.f / kHid);
    else if (i >= kOffW3 && i < kOffB3) v = u * sqrtf(6.f / kHid);
    p[i] = v;
  }
}

// x[b][j] = registers[b * stride + j] / 64: sketch registers as network inputs.
__global__ void k_features(const uint32_t *regs, int64_t stride, int B, float *x) {
  after_previous();
  const int64_t n = (int64_t)B * kIn;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x)
    x[i] = (float)regs[(i / kIn) * stride + (i % kIn)] * (1.0f / 64.0f);
}

Work carve(float *w, int B) {
  Work k;
  k.h1 = w;
  k.h2 = k.h1 + (size_t)B * kHid;
  k.dh1 = k.h2 + (size_t)B * kHid;
  k.dh2 = k.dh1 + (size_t)B * kHid;
  k.y = k.dh2 + (size_t)B * kHid;
  k.dy = k.y + B;
  k.loss = k.dy + B;
  return k;
}

}  // namespace
}  // namespace dbg

using namespace dbg;

extern "C" uint64_t dbg_mlp_work_floats(int batch) {
  return batch <= 0 ? 0 : (uint64_t)batch * (4 * DBG_MLP_HIDDEN + 2) + 1;
}

extern "C" int dbg_mlp_features(const uint32_t *registers, int64_t stride, int batch, float *x,
                                void *stream) {
  if (!registers || !x || batch <= 0 || stride < DBG_MLP_INPUTS) return DBG_ERR_INVALID_ARG;
  DBG_TRY(launch_after(k_features, 256, 256, 0, static_cast<cudaStream_t>(stream), registers,
                       stride, batch, x));
  DBG_CK(cudaGetLastError());
  return DBG_OK;
}

extern "C" int dbg_mlp_init(float *params, uint64_t seed, void *stream) {
  if (!params) return DBG_ERR_INVALID_ARG;
  k_init<<<64, 256, 0, static_cast<cudaStream_t>(stream)>>>(params, seed);
  DBG_CK(cudaGetLastError());
  return DBG_OK;
}

extern "C" int dbg_mlp_forward(const float *params, const float *x, int batch, float *y,
                               float *work, void *stream) {
  if (!params || !x || !y || !work || batch <= 0) return DBG_ERR_INVALID_ARG;
  DBG_TRY(launch_after(k_rows<false>, (batch + kRows - 1) / kRows, 32 * kWarps, 0,
                       static_cast<cudaStream_t>(stream), params, x, nullptr, batch, y, Work{}));
  DBG_CK(cudaGetLastError());
  return DBG_OK;
}

extern "C" int dbg_mlp_train_step(float *params, float *grads, float *adam_m, float *adam_v,
                                  int step, float lr, const float *x, const float *target,
                                  int batch, float *work, float *loss_out, void *stream) {
  if (!params || !grads || !adam_m || !adam_v || !x || !target || !work || batch <= 0 ||
      step < 1 || !(lr > 0.f))
    return DBG_ERR_INVALID_ARG;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  const Work w = carve(work, batch);
  DBG_TRY(launch_after(k_rows<true>, (batch + kRows - 1) / kRows, 32 * kWarps, 0, s, params, x,
                       target, batch, w.y, w));
  DBG_CK(cudaGetLastError());
  const float b1 = 0.9f, b2 = 0.999f;
  const Adam ad{params, grads, adam_m, adam_v, lr,
                b1,     b2,    1e-8f,  1.f - powf(b1, (float)step), 1.f - powf(b2, (float)step)};
  DBG_TRY(launch_after(k_grads, kGradCtas, 256, 0, s, x, target, batch, w, ad));
  DBG_CK(cudaGetLastError());
  if (loss_out) DBG_CK(cudaMemcpyAsync(loss_out, w.loss, sizeof(float), cudaMemcpyDefault, s));
  return DBG_OK;
}
