// K8/K9: the learned row-size predictor (paper Sec. 5: the GPU path estimates
// the output's memory needs with approximate algorithms instead of an exact
// symbolic pass; Sec. 7.4: the batch count of batched SpGEMM comes from
// such an estimate).
//
// Model: 3 -> 64 -> 64 -> 1 MLP over the row features f = (nnz(A_i), flops_i,
// max_p nnz(B_p)), the last two taken relative to the row's output width w_i
// (the column count of B), so that the same network serves products of any
// size:
//   l  = (log2(1 + f_0), log2(1 + f_1) - log2(w_i), log2(1 + f_2) - log2(w_i))
//   x  = bf16((l - mu) / sigma)
//   h1 = bf16(relu(W1 x + b1)),  h2 = bf16(relu(W2 h1 + b2)),  z = w3 . h2 + b3
//   rho = sigmoid(z) ~ nnz(C_i) / flops_i,
//   pred = clamp(ceil(rho * flops_i), maxB_i, min(flops_i, w_i))
// Feature rows are float32 [4]: nnz(A_i), flops_i, maxB_i, w_i.
// Weights are used as bf16 copies of fp32 master weights; every product is
// accumulated in fp32.  Training minimises the pinball loss (tau) on
// e = log2(nnz/flops) - log2(rho) with Adam on the fp32 master weights.
#include <cuda_bf16.h>

#include <cmath>
#include <cstring>
#include <new>
#include <string>

#include "../../include/cb.h"
#include "cb_common.cuh"

namespace cb {
namespace {

constexpr int H = CB_MLP_HIDDEN;
// offsets into the flat parameter vector
constexpr int oW1 = 0, ob1 = oW1 + H * 3, oW2 = ob1 + H, ob2 = oW2 + H * H, ow3 = ob2 + H,
              ob3 = ow3 + H, kNP = ob3 + 1;
static_assert(kNP == CB_MLP_NPARAM, "parameter layout");

constexpr int kFwdThreads = 256;
constexpr int kBatchUnit = 128;  // training batches are rounded up to a multiple of this

__device__ __forceinline__ float bf16r(float v) { return __bfloat162float(__float2bfloat16_rn(v)); }

constexpr int kNF = CB_MLP_NFEAT;  // floats per feature row

// The small weights, staged in shared memory (bf16 values held as floats).
struct SmallWeights {
  float4 w1b[H];  // W1 row j and b1[j]
  float b2[H], w3[H], b3, mu[3], sg[3];
};

__device__ __forceinline__ void stage_small(SmallWeights& w, const __nv_bfloat16* wb, const float* master,
                                            const float* norm) {
  for (int t = threadIdx.x; t < H; t += blockDim.x) {
    w.w1b[t] = make_float4(__bfloat162float(wb[oW1 + 3 * t]), __bfloat162float(wb[oW1 + 3 * t + 1]),
                           __bfloat162float(wb[oW1 + 3 * t + 2]), master[ob1 + t]);
    w.b2[t] = master[ob2 + t];
    w.w3[t] = __bfloat162float(wb[ow3 + t]);
  }
  if (threadIdx.x == 0) w.b3 = master[ob3];
  if (threadIdx.x < 3) {
    w.mu[threadIdx.x] = norm[threadIdx.x];
    w.sg[threadIdx.x] = norm[3 + threadIdx.x];
  }
}

__device__ __forceinline__ void features(const SmallWeights& w, const float* f, float x[3]) {
  const float lw = log2f(fmaxf(f[3], 1.0f));
  float l[3] = {log2f(1.0f + f[0]), log2f(1.0f + f[1]) - lw, log2f(1.0f + f[2]) - lw};
#pragma unroll
  for (int d = 0; d < 3; ++d) x[d] = bf16r((l[d] - w.mu[d]) / w.sg[d]);
}

// h1[j] of one row.
__device__ __forceinline__ float hidden1(const SmallWeights& w, int j, const float x[3]) {
  const float4 v = w.w1b[j];
  float a = v.w;
  a = fmaf(v.x, x[0], a);
  a = fmaf(v.y, x[1], a);
  a = fmaf(v.z, x[2], a);
  return bf16r(fmaxf(a, 0.0f));
}

__device__ __forceinline__ int64_t size_from_logit(float z, int64_t flops, int64_t maxb,
                                                   int64_t width, int64_t ncols) {
  if (flops <= 0) return 0;
  const double rho = 1.0 / (1.0 + exp(-(double)z));
  int64_t est = (int64_t)ceil(rho * (double)flops);
  int64_t hi = flops < width ? flops : width;
  if (ncols > 0 && ncols < hi) hi = ncols;
  if (est < maxb) est = maxb;
  if (est > hi) est = hi;
  return est;
}

// K8: a warp per 32 rows.  Every sum runs over its inputs in ascending order
// in fp32 (one rounding per product), whichever thread holds it, so logits do
// not depend on the layout.  The 64 x 64 layer is an outer-product loop on
// 8 rows x 8 outputs per lane: h1 lies [input][row] in shared memory, W2
// transposed, and each step of 64 FMAs per lane reads four 16-byte vectors
// (shared-memory bandwidth and FMA issue are about even; one thread per row,
// which read two shared words per FMA, took 379 us for 524288 rows).
constexpr int kFwdWarps = kFwdThreads / 32;
constexpr int kRowPad = H + 4;  // row stride of h2: 16-byte reads of 8 rows meet all banks
struct PredictSmem {
  SmallWeights s;
  float w2t[H * H];                    // [input][output]
  float h[kFwdWarps][32 * kRowPad];    // a warp's h1 [input][32 rows], then h2 [row][kRowPad]
};

__global__ void __launch_bounds__(kFwdThreads, 2) k_mlp_predict(const __nv_bfloat16* wb, const float* master,
                                                                const float* norm, const float* feat,
                                                                int64_t m, int64_t ncols, float* z_out,
                                                                int64_t* pred_out) {
  extern __shared__ __align__(16) unsigned char mlp_smem[];
  PredictSmem& w = *reinterpret_cast<PredictSmem*>(mlp_smem);
  stage_small(w.s, wb, master, norm);
  for (int t = threadIdx.x; t < H * H; t += kFwdThreads)
    w.w2t[(t % H) * H + t / H] = __bfloat162float(wb[oW2 + t]);
  __syncthreads();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int rg = lane >> 3, jg = lane & 7;  // rows 8 rg .. + 7, outputs 4 jg .. + 3 and 32 + 4 jg .. + 3
  float* const h = w.h[warp];
  for (int64_t r0 = ((int64_t)blockIdx.x * kFwdWarps + warp) * 32; r0 < m;
       r0 += (int64_t)gridDim.x * kFwdThreads) {
    const int64_t r = r0 + lane;
    float f[kNF] = {0.0f, 0.0f, 0.0f, 1.0f}, x[3];
    if (r < m) {
#pragma unroll
      for (int d = 0; d < kNF; ++d) f[d] = feat[kNF * r + d];
    }
    features(w.s, f, x);
#pragma unroll 4
    for (int j = 0; j < H; ++j) h[32 * j + lane] = hidden1(w.s, j, x);
    __syncwarp();
    float acc[8][8];  // [row][output]
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const float b = w.s.b2[(q < 4 ? 0 : 28) + 4 * jg + q];
#pragma unroll
      for (int i = 0; i < 8; ++i) acc[i][q] = b;
    }
#pragma unroll 2
    for (int k = 0; k < H; ++k) {
      float a[8], b[8];
      *reinterpret_cast<float4*>(a) = *reinterpret_cast<const float4*>(h + 32 * k + 8 * rg);
      *reinterpret_cast<float4*>(a + 4) = *reinterpret_cast<const float4*>(h + 32 * k + 8 * rg + 4);
      *reinterpret_cast<float4*>(b) = *reinterpret_cast<const float4*>(w.w2t + H * k + 4 * jg);
      *reinterpret_cast<float4*>(b + 4) = *reinterpret_cast<const float4*>(w.w2t + H * k + 32 + 4 * jg);
#pragma unroll
      for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int q = 0; q < 8; ++q) acc[i][q] = fmaf(b[q], a[i], acc[i][q]);
    }
    __syncwarp();  // h1 is read; h2 takes its place
#pragma unroll
    for (int i = 0; i < 8; ++i) {
#pragma unroll
      for (int q = 0; q < 8; ++q) acc[i][q] = bf16r(fmaxf(acc[i][q], 0.0f));
      float* const o = h + (8 * rg + i) * kRowPad + 4 * jg;
      *reinterpret_cast<float4*>(o) = make_float4(acc[i][0], acc[i][1], acc[i][2], acc[i][3]);
      *reinterpret_cast<float4*>(o + 32) = make_float4(acc[i][4], acc[i][5], acc[i][6], acc[i][7]);
    }
    __syncwarp();
    float z = w.s.b3;
#pragma unroll
    for (int j = 0; j < H; j += 4) {
      const float4 v = *reinterpret_cast<const float4*>(h + lane * kRowPad + j);
      z = fmaf(w.s.w3[j], v.x, z);
      z = fmaf(w.s.w3[j + 1], v.y, z);
      z = fmaf(w.s.w3[j + 2], v.z, z);
      z = fmaf(w.s.w3[j + 3], v.w, z);
    }
    if (r < m) {
      if (z_out) z_out[r] = z;
      if (pred_out) pred_out[r] = size_from_logit(z, (int64_t)f[1], (int64_t)f[2], (int64_t)f[3], ncols);
    }
    __syncwarp();  // h2 is read; the next rows' h1 takes its place
  }
}

// K9: forward + pinball loss + backward for rows [r0, r0 + n).  Gradient sums
// (not yet divided by the number of live rows) are added to grad[0..kNP),
// the loss sum to stat[0] and the live-row count to stat[1].
// A CTA takes 64 rows at a time: both 64 x 64 x 64 products of the layer (and
// the third, its weight gradient) run on 4 x 4 outputs per thread from
// shared-memory tiles [unit][row], and the weight gradient stays in registers
// until the CTA's last rows.  8192 rows, a training mini-batch, then run on
// 128 SMs at once.  (128 rows per 128-thread CTA, a row per thread with its
// layer loops serial, kept 64 SMs busy for 94 us.)
constexpr int kBwdRows = 64, kBwdThreads = 256;
constexpr int kTile = kBwdRows + 4;  // row stride of the tiles
struct GradSmem {
  SmallWeights s;
  float w2[H * H], w2t[H * H];   // [output][input], [input][output]
  float h1[H * kTile], d2[H * kTile], d1[H * kTile];  // [unit][row]; d2 holds h2 first
  float x[3][kBwdRows], dz[kBwdRows];
};

__global__ void __launch_bounds__(kBwdThreads) k_mlp_grad(const __nv_bfloat16* wb, const float* master,
                                                          const float* norm, const float* feat,
                                                          const int64_t* nnz, int64_t r0, int64_t n, float tau,
                                                          float* grad, double* stat) {
  extern __shared__ __align__(16) unsigned char mlp_smem[];
  GradSmem& w = *reinterpret_cast<GradSmem*>(mlp_smem);
  stage_small(w.s, wb, master, norm);
  for (int t = threadIdx.x; t < H * H; t += kBwdThreads) {
    const float v = __bfloat162float(wb[oW2 + t]);
    w.w2[t] = v;
    w.w2t[(t % H) * H + t / H] = v;
  }
  const int tid = threadIdx.x;
  const int lo4 = 4 * (tid & 15), hi4 = 4 * (tid >> 4);  // 4 x 4 tile: rows (or inputs), units
  const int unit = tid >> 2, part = tid & 3;             // sums over 16 rows of one unit
  float gw2[4][4] = {};                                  // [output hi4 + a][input tid % 16 + 16 b]
  float gw3 = 0.0f, gb2 = 0.0f, gb1 = 0.0f, gw1[3] = {0.0f, 0.0f, 0.0f}, gb3 = 0.0f;
  double loss_sum = 0.0;
  int live_sum = 0;
  for (int64_t base = (int64_t)blockIdx.x * kBwdRows; base < n; base += (int64_t)gridDim.x * kBwdRows) {
    __syncthreads();  // weights staged; the last tile's readers are done
    {
      const int row = tid & (kBwdRows - 1), j0 = (tid / kBwdRows) * 16;
      const int64_t r = base + row;
      float x[3] = {0.0f, 0.0f, 0.0f};
      if (r < n) features(w.s, feat + kNF * (r0 + r), x);
#pragma unroll 4
      for (int j = j0; j < j0 + 16; ++j) w.h1[j * kTile + row] = r < n ? hidden1(w.s, j, x) : 0.0f;
      if (tid < kBwdRows) {
        w.x[0][row] = x[0];
        w.x[1][row] = x[1];
        w.x[2][row] = x[2];
      }
    }
    __syncthreads();
    {  // h2[hi4 + b][lo4 + a]
      float acc[4][4];
#pragma unroll
      for (int b = 0; b < 4; ++b)
#pragma unroll
        for (int a = 0; a < 4; ++a) acc[b][a] = w.s.b2[hi4 + b];
#pragma unroll 4
      for (int k = 0; k < H; ++k) {
        float h[4], v[4];
        *reinterpret_cast<float4*>(h) = *reinterpret_cast<const float4*>(w.h1 + k * kTile + lo4);
        *reinterpret_cast<float4*>(v) = *reinterpret_cast<const float4*>(w.w2t + k * H + hi4);
#pragma unroll
        for (int b = 0; b < 4; ++b)
#pragma unroll
          for (int a = 0; a < 4; ++a) acc[b][a] = fmaf(v[b], h[a], acc[b][a]);
      }
#pragma unroll
      for (int b = 0; b < 4; ++b)
        *reinterpret_cast<float4*>(w.d2 + (hi4 + b) * kTile + lo4) =
            make_float4(bf16r(fmaxf(acc[b][0], 0.0f)), bf16r(fmaxf(acc[b][1], 0.0f)),
                        bf16r(fmaxf(acc[b][2], 0.0f)), bf16r(fmaxf(acc[b][3], 0.0f)));
    }
    __syncthreads();
    if (tid < kBwdRows) {  // the logit, its loss and slope
      float z = w.s.b3;
#pragma unroll 8
      for (int j = 0; j < H; ++j) z = fmaf(w.s.w3[j], w.d2[j * kTile + tid], z);
      float dz = 0.0f;
      const int64_t r = base + tid;
      if (r < n) {
        const float fl = feat[kNF * (r0 + r) + 1];
        if (fl > 0.0f) {
          const float ls = -(fmaxf(-z, 0.0f) + log1pf(expf(-fabsf(z))));  // log sigmoid(z)
          const float e = log2f((float)nnz[r0 + r] / fl) - ls * 1.4426950408889634f;
          loss_sum += (double)(e >= 0.0f ? tau * e : (tau - 1.0f) * e);
          ++live_sum;
          const float sig = 1.0f / (1.0f + expf(-z));
          dz = (e >= 0.0f ? tau : tau - 1.0f) * (-(1.0f - sig) * 1.4426950408889634f);
        }
      }
      w.dz[tid] = dz;
      gb3 += dz;
    }
    __syncthreads();
    {  // h2 -> its gradient in place, with the sums that need it
      const float w3 = w.s.w3[unit];
#pragma unroll 4
      for (int t = 0; t < 16; ++t) {
        const int row = 16 * part + t;
        float* const p = w.d2 + unit * kTile + row;
        const float h = *p, dz = w.dz[row];
        gw3 = fmaf(dz, h, gw3);
        const float d = h > 0.0f ? dz * w3 : 0.0f;
        gb2 += d;
        *p = d;
      }
    }
    __syncthreads();
    {  // d1[hi4 + b][lo4 + a], and the weight gradient's outer products
      float acc[4][4] = {};
#pragma unroll 4
      for (int j = 0; j < H; ++j) {
        float d[4], v[4];
        *reinterpret_cast<float4*>(d) = *reinterpret_cast<const float4*>(w.d2 + j * kTile + lo4);
        *reinterpret_cast<float4*>(v) = *reinterpret_cast<const float4*>(w.w2 + j * H + hi4);
#pragma unroll
        for (int b = 0; b < 4; ++b)
#pragma unroll
          for (int a = 0; a < 4; ++a) acc[b][a] = fmaf(d[a], v[b], acc[b][a]);
      }
#pragma unroll
      for (int b = 0; b < 4; ++b) {
        const float4 h = *reinterpret_cast<const float4*>(w.h1 + (hi4 + b) * kTile + lo4);
        *reinterpret_cast<float4*>(w.d1 + (hi4 + b) * kTile + lo4) =
            make_float4(h.x > 0.0f ? acc[b][0] : 0.0f, h.y > 0.0f ? acc[b][1] : 0.0f,
                        h.z > 0.0f ? acc[b][2] : 0.0f, h.w > 0.0f ? acc[b][3] : 0.0f);
      }
#pragma unroll 2
      for (int r = 0; r < kBwdRows; r += 4) {
        float4 d[4], h[4];
#pragma unroll
        for (int a = 0; a < 4; ++a) d[a] = *reinterpret_cast<const float4*>(w.d2 + (hi4 + a) * kTile + r);
#pragma unroll
        for (int b = 0; b < 4; ++b)
          h[b] = *reinterpret_cast<const float4*>(w.h1 + ((tid & 15) + 16 * b) * kTile + r);
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
          for (int b = 0; b < 4; ++b) {
            gw2[a][b] = fmaf(d[a].x, h[b].x, gw2[a][b]);
            gw2[a][b] = fmaf(d[a].y, h[b].y, gw2[a][b]);
            gw2[a][b] = fmaf(d[a].z, h[b].z, gw2[a][b]);
            gw2[a][b] = fmaf(d[a].w, h[b].w, gw2[a][b]);
          }
      }
    }
    __syncthreads();
#pragma unroll 4
    for (int t = 0; t < 16; ++t) {
      const int row = 16 * part + t;
      const float d = w.d1[unit * kTile + row];
      gb1 += d;
      gw1[0] = fmaf(d, w.x[0][row], gw1[0]);
      gw1[1] = fmaf(d, w.x[1][row], gw1[1]);
      gw1[2] = fmaf(d, w.x[2][row], gw1[2]);
    }
  }
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int b = 0; b < 4; ++b) atomicAdd(&grad[oW2 + (hi4 + a) * H + (tid & 15) + 16 * b], gw2[a][b]);
  float sums[6] = {gw3, gb2, gb1, gw1[0], gw1[1], gw1[2]};
#pragma unroll
  for (int q = 0; q < 6; ++q) {
    sums[q] += __shfl_xor_sync(0xffffffffu, sums[q], 1);
    sums[q] += __shfl_xor_sync(0xffffffffu, sums[q], 2);
  }
  if (part == 0) {
    atomicAdd(&grad[ow3 + unit], sums[0]);
    atomicAdd(&grad[ob2 + unit], sums[1]);
    atomicAdd(&grad[ob1 + unit], sums[2]);
    atomicAdd(&grad[oW1 + unit * 3 + 0], sums[3]);
    atomicAdd(&grad[oW1 + unit * 3 + 1], sums[4]);
    atomicAdd(&grad[oW1 + unit * 3 + 2], sums[5]);
  }
  if (tid < kBwdRows) {
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) {
      gb3 += __shfl_down_sync(0xffffffffu, gb3, d);
      loss_sum += __shfl_down_sync(0xffffffffu, loss_sum, d);
      live_sum += __shfl_down_sync(0xffffffffu, live_sum, d);
    }
    if ((tid & 31) == 0) {
      atomicAdd(&grad[ob3], gb3);
      atomicAdd(&stat[0], loss_sum);
      atomicAdd(&stat[1], (double)live_sum);
    }
  }
}

// Divide gradient sums by the live-row count (gradient output form).
__global__ void k_mlp_scale(const float* grad, const double* stat, float* out, float* loss) {
  const double inv = stat[1] > 0 ? 1.0 / stat[1] : 0.0;
  for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < kNP; t += gridDim.x * blockDim.x)
    out[t] = (float)(grad[t] * inv);
  if (blockIdx.x == 0 && threadIdx.x == 0 && loss) *loss = (float)(stat[0] * inv);
}

// Adam step on the master weights with the mean gradient, refresh the bf16
// copies, clear the gradient sums and the batch statistics.  One block (it
// clears the statistics that all threads read first).
__global__ void k_mlp_adam(float* master, __nv_bfloat16* wb, float* mom, float* vel, float* grad,
                           double* stat, double* epoch_loss, float lr, float b1c, float b2c,
                           int64_t step) {
  const double live = stat[1];
  const float inv = live > 0 ? (float)(1.0 / live) : 0.0f;
  const float c1 = 1.0f - powf(b1c, (float)step), c2 = 1.0f - powf(b2c, (float)step);
  for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < kNP; t += gridDim.x * blockDim.x) {
    const float g = grad[t] * inv;
    const float mt = b1c * mom[t] + (1.0f - b1c) * g;
    const float vt = b2c * vel[t] + (1.0f - b2c) * g * g;
    mom[t] = mt;
    vel[t] = vt;
    const float wnew = master[t] - lr * (mt / c1) / (sqrtf(vt / c2) + 1e-8f);
    master[t] = wnew;
    wb[t] = __float2bfloat16_rn(wnew);
    grad[t] = 0.0f;
  }
  __syncthreads();
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    if (epoch_loss) {
      epoch_loss[0] += stat[0];
      epoch_loss[1] += stat[1];
    }
    stat[0] = 0.0;
    stat[1] = 0.0;
  }
}

__global__ void k_mlp_round(const float* master, __nv_bfloat16* wb) {
  for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < kNP; t += gridDim.x * blockDim.x)
    wb[t] = __float2bfloat16_rn(master[t]);
}

// raw features (nnz(A_i), flops_i, maxB_i) as floats
__global__ void k_row_features(DevCSR A, const int64_t* flops, const int32_t* maxb, int64_t ncols,
                               float* feat) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < A.nrows;
       i += (int64_t)gridDim.x * blockDim.x) {
    feat[kNF * i + 0] = (float)(A.rp[i + 1] - A.rp[i]);
    feat[kNF * i + 1] = (float)flops[i];
    feat[kNF * i + 2] = (float)maxb[i];
    feat[kNF * i + 3] = (float)(A.rcols ? (int64_t)A.rcols[i] : ncols);
  }
}

// Launch over n rows; the shared-memory limit is the current device's.
void run_grad(const __nv_bfloat16* wb, const float* master, const float* norm, const float* feat,
              const int64_t* nnz, int64_t r0, int64_t n, float tau, float* grad, double* stat, int sms,
              cudaStream_t s) {
  cudaFuncSetAttribute(k_mlp_grad, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(GradSmem));
  const int64_t tiles = (n + kBwdRows - 1) / kBwdRows, most = 2 * (int64_t)sms;
  k_mlp_grad<<<(unsigned)(tiles < most ? tiles : most), kBwdThreads, sizeof(GradSmem), s>>>(
      wb, master, norm, feat, nnz, r0, n, tau, grad, stat);
}

}  // namespace

void launch_row_features(const DevCSR& A, const int64_t* flops, const int32_t* maxb, int64_t ncols,
                         float* feat, cudaStream_t s, int sms) {
  if (A.nrows == 0) return;
  int64_t g = (A.nrows + 255) / 256;
  k_row_features<<<(int)(g < sms * 8 ? g : sms * 8), 256, 0, s>>>(A, flops, maxb, ncols, feat);
}

void launch_mlp_predict(const void* wb, const float* master, const float* norm, const float* feat,
                        int64_t m, int64_t ncols, float* z, int64_t* pred, cudaStream_t s, int sms) {
  if (m == 0) return;
  cudaFuncSetAttribute(k_mlp_predict, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(PredictSmem));
  const int64_t g = (m + kFwdThreads - 1) / kFwdThreads;
  k_mlp_predict<<<(int)(g < sms * 2 ? g : sms * 2), kFwdThreads, sizeof(PredictSmem), s>>>(
      static_cast<const __nv_bfloat16*>(wb), master, norm, feat, m, ncols, z, pred);
}

}  // namespace cb

// ---------------------------------------------------------------------------
// C ABI
// ---------------------------------------------------------------------------

struct cb_mlp {
  int device = 0;
  float* master = nullptr;     // kNP fp32
  __nv_bfloat16* wb = nullptr; // kNP bf16 copies
  float* mom = nullptr;
  float* vel = nullptr;
  float* grad = nullptr;
  float* norm = nullptr;       // mu[3], sigma[3]
  double* stat = nullptr;      // loss sum, live rows; then epoch loss sum, epoch live rows
  int64_t step = 0;
};

namespace {
int mlp_free(cb_mlp* m) {
  if (!m) return CB_OK;
  cudaFree(m->master);
  cudaFree(m->wb);
  cudaFree(m->mom);
  cudaFree(m->vel);
  cudaFree(m->grad);
  cudaFree(m->norm);
  cudaFree(m->stat);
  delete m;
  return CB_OK;
}
}  // namespace

extern "C" {

int cb_mlp_create(cb_mlp** out, const float* params, const float* norm) {
  using namespace cb;
  if (!out || !params || !norm) return CB_ERR_ARG;
  *out = nullptr;
  cb_mlp* m = new (std::nothrow) cb_mlp();
  if (!m) return CB_ERR_OOM;
  cudaGetDevice(&m->device);
  bool ok = cudaMalloc(&m->master, kNP * sizeof(float)) == cudaSuccess &&
            cudaMalloc(&m->wb, kNP * sizeof(__nv_bfloat16)) == cudaSuccess &&
            cudaMalloc(&m->mom, kNP * sizeof(float)) == cudaSuccess &&
            cudaMalloc(&m->vel, kNP * sizeof(float)) == cudaSuccess &&
            cudaMalloc(&m->grad, kNP * sizeof(float)) == cudaSuccess &&
            cudaMalloc(&m->norm, 6 * sizeof(float)) == cudaSuccess &&
            cudaMalloc(&m->stat, 4 * sizeof(double)) == cudaSuccess;
  if (!ok) {
    mlp_free(m);
    return CB_ERR_OOM;
  }
  ok = cudaMemcpy(m->master, params, kNP * sizeof(float), cudaMemcpyHostToDevice) == cudaSuccess &&
       cudaMemcpy(m->norm, norm, 6 * sizeof(float), cudaMemcpyHostToDevice) == cudaSuccess &&
       cudaMemset(m->mom, 0, kNP * sizeof(float)) == cudaSuccess &&
       cudaMemset(m->vel, 0, kNP * sizeof(float)) == cudaSuccess &&
       cudaMemset(m->grad, 0, kNP * sizeof(float)) == cudaSuccess &&
       cudaMemset(m->stat, 0, 4 * sizeof(double)) == cudaSuccess;
  if (ok) {
    k_mlp_round<<<8, 256>>>(m->master, m->wb);
    ok = cudaGetLastError() == cudaSuccess && cudaDeviceSynchronize() == cudaSuccess;
  }
  if (!ok) {
    mlp_free(m);
    return CB_ERR_CUDA;
  }
  *out = m;
  return CB_OK;
}

void cb_mlp_destroy(cb_mlp* m) {
  if (m) cudaDeviceSynchronize();
  mlp_free(m);
}

int cb_mlp_get(const cb_mlp* m, float* params, float* norm, int64_t* step) {
  using namespace cb;
  if (!m) return CB_ERR_ARG;
  if (cudaDeviceSynchronize() != cudaSuccess) return CB_ERR_CUDA;
  if (params && cudaMemcpy(params, m->master, kNP * sizeof(float), cudaMemcpyDeviceToHost) != cudaSuccess)
    return CB_ERR_CUDA;
  if (norm && cudaMemcpy(norm, m->norm, 6 * sizeof(float), cudaMemcpyDeviceToHost) != cudaSuccess)
    return CB_ERR_CUDA;
  if (step) *step = m->step;
  return CB_OK;
}

}  // extern "C"

// Device-side accessors used by the SpGEMM dispatcher (learned sizing).
namespace cb {
const void* mlp_bf16(const cb_mlp* m) { return m->wb; }
const float* mlp_master(const cb_mlp* m) { return m->master; }
const float* mlp_norm(const cb_mlp* m) { return m->norm; }
}  // namespace cb

extern "C" {

int cb_mlp_predict(cb_ctx* ctx, const cb_mlp* m, const float* feat, int64_t nrows, int64_t ncols,
                   float* z, int64_t* pred);
int cb_mlp_grad(cb_ctx* ctx, const cb_mlp* m, const float* feat, const int64_t* nnz, int64_t nrows,
                float tau, float* grad, float* loss);
int cb_mlp_train(cb_ctx* ctx, cb_mlp* m, const float* feat, const int64_t* nnz, int64_t nrows,
                 int epochs, int64_t batch, float lr, float tau, float* epoch_loss);

}  // extern "C"

// Shared with the context-owning file.
namespace cb {
cudaStream_t ctx_stream(cb_ctx* ctx);
int ctx_sms(cb_ctx* ctx);
}  // namespace cb

extern "C" int cb_mlp_predict(cb_ctx* ctx, const cb_mlp* m, const float* feat, int64_t nrows,
                              int64_t ncols, float* z, int64_t* pred) {
  if (!ctx || !m || nrows < 0 || (nrows > 0 && !feat) || ncols < 0) return CB_ERR_ARG;
  cb::launch_mlp_predict(m->wb, m->master, m->norm, feat, nrows, ncols, z, pred, cb::ctx_stream(ctx),
                         cb::ctx_sms(ctx));
  return cudaGetLastError() == cudaSuccess ? CB_OK : CB_ERR_CUDA;
}

extern "C" int cb_mlp_grad(cb_ctx* ctx, const cb_mlp* m, const float* feat, const int64_t* nnz,
                           int64_t nrows, float tau, float* grad, float* loss) {
  using namespace cb;
  if (!ctx || !m || nrows < 0 || (nrows > 0 && (!feat || !nnz)) || !grad) return CB_ERR_ARG;
  cudaStream_t s = ctx_stream(ctx);
  if (cudaMemsetAsync(m->grad, 0, kNP * sizeof(float), s) != cudaSuccess ||
      cudaMemsetAsync(m->stat, 0, 2 * sizeof(double), s) != cudaSuccess)
    return CB_ERR_CUDA;
  if (nrows > 0)
    run_grad(m->wb, m->master, m->norm, feat, nnz, 0, nrows, tau, m->grad, m->stat, ctx_sms(ctx), s);
  k_mlp_scale<<<8, 256, 0, s>>>(m->grad, m->stat, grad, loss);
  const bool ok = cudaGetLastError() == cudaSuccess &&
                  cudaMemsetAsync(m->grad, 0, kNP * sizeof(float), s) == cudaSuccess &&
                  cudaMemsetAsync(m->stat, 0, 2 * sizeof(double), s) == cudaSuccess;
  return ok ? CB_OK : CB_ERR_CUDA;
}

extern "C" int cb_mlp_train(cb_ctx* ctx, cb_mlp* m, const float* feat, const int64_t* nnz,
                            int64_t nrows, int epochs, int64_t batch, float lr, float tau,
                            float* epoch_loss) {
  using namespace cb;
  if (!ctx || !m || nrows <= 0 || !feat || !nnz || epochs < 0 || batch <= 0 || !(lr > 0.0f))
    return CB_ERR_ARG;
  cudaStream_t s = ctx_stream(ctx);
  if (batch % kBatchUnit) batch += kBatchUnit - batch % kBatchUnit;
  if (cudaMemsetAsync(m->grad, 0, kNP * sizeof(float), s) != cudaSuccess ||
      cudaMemsetAsync(m->stat, 0, 4 * sizeof(double), s) != cudaSuccess)
    return CB_ERR_CUDA;
  for (int ep = 0; ep < epochs; ++ep) {
    // each epoch starts the batch sequence at a different offset
    const int64_t shift = ((int64_t)ep * 7919 * kBatchUnit) % nrows;
    for (int64_t done = 0; done < nrows; done += batch) {
      const int64_t start = (shift + done) % nrows;
      int64_t n = batch < nrows - done ? batch : nrows - done;
      // a batch that runs past the end wraps to the front in two launches
      const int64_t n1 = n < nrows - start ? n : nrows - start;
      run_grad(m->wb, m->master, m->norm, feat, nnz, start, n1, tau, m->grad, m->stat, ctx_sms(ctx), s);
      if (n > n1)
        run_grad(m->wb, m->master, m->norm, feat, nnz, 0, n - n1, tau, m->grad, m->stat, ctx_sms(ctx), s);
      ++m->step;
      k_mlp_adam<<<1, 1024, 0, s>>>(m->master, m->wb, m->mom, m->vel, m->grad, m->stat,
                                    m->stat + 2, lr, 0.9f, 0.999f, m->step);
    }
    if (epoch_loss) {
      double h[2];
      if (cudaMemcpyAsync(h, m->stat + 2, 2 * sizeof(double), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
          cudaStreamSynchronize(s) != cudaSuccess ||
          cudaMemsetAsync(m->stat + 2, 0, 2 * sizeof(double), s) != cudaSuccess)
        return CB_ERR_CUDA;
      epoch_loss[ep] = h[1] > 0 ? (float)(h[0] / h[1]) : 0.0f;
    }
  }
  return cudaGetLastError() == cudaSuccess ? CB_OK : CB_ERR_CUDA;
}
