// Cost-model network: fp32 multilayer perceptron that predicts a variant's
// log run time (a per-query variant choice, the run-time optimizer the paper
// leaves to future work, Section 9.4).
//
//   xh = (x - mu) / sigma            F features
//   z1 = xh W1 + b1, h1 = relu(z1)   H = 64 units
//   z2 = h1 W2 + b2, h2 = relu(z2)   H units
//   y  = h2 w3 + b3
//   L  = mean over the batch of (y - t)^2
//
// Parameters are one float vector: W1 (F x H, row-major), b1, W2 (H x H),
// b2, w3, b3.  Adam (Kingma and Ba, 2015, Algorithm 1) updates it in place.
// The products are small fp32 matrix products, done by tiles of samples on
// the FMA units (fp32 in, fp32 accumulate): a CTA stages a tile's operands in
// shared memory and each of its 256 threads keeps a block of 4 x 4 (samples x
// units, or inputs x units for the weight gradients) in registers, so that two
// 16-byte shared loads feed 16 FMAs.  One sample per thread with the weights
// read as broadcasts gave an SM five warps and every FMA its own shared
// operand: 77 us forward and 63 + 68 us backward for 24,001 samples of 45
// features, against 12 us of FMAs (a whole training step 190 us, now 59 us).
#include <algorithm>

#include <cstdint>

#include "pv_internal.h"

namespace pv {

constexpr int kH = PV_MLP_HIDDEN;
constexpr int kMaxF = PV_MLP_MAX_FEATURES;
constexpr int kMlpBlock = 256;  // 16 x 16 threads
constexpr int kTile = 64;       // samples per CTA, forward
constexpr int kLd = kH + 4;     // leading dimension of transposed tiles: rows stay 16-byte aligned

struct MlpArgs {
  const float* p;      // parameters
  const float* x;      // [B x F]
  const float* mu;     // [F]
  const float* sigma;  // [F]
  float* y;            // [B]
  float* act;          // [B x 2H]: z1 then z2 of every sample (may be null in forward)
  const float* t;      // [B] targets
  float* grad;         // same layout as p; backward: copy r at grad + r * stride
  float* loss;         // [1]; backward: copy r at loss + r * stride
  int copies;          // of the gradient and the loss the CTAs add into
  int64_t stride;
  int B, F;
};

__host__ __device__ inline int64_t mlp_n_params(int F) { return static_cast<int64_t>(F) * kH + kH + kH * kH + kH + kH + 1; }

__device__ __forceinline__ bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

__device__ __forceinline__ float4 ld4(const float* p, bool vec) {
  if (vec) return *reinterpret_cast<const float4*>(p);
  return make_float4(p[0], p[1], p[2], p[3]);
}
__device__ __forceinline__ float4 lds4(const float* p) { return *reinterpret_cast<const float4*>(p); }

// n floats of global memory into shared memory (16-byte aligned there).
__device__ __forceinline__ void stage_floats(float* d, const float* g, int n) {
  int i = 0;
  if (aligned16(g)) {
    for (i = threadIdx.x * 4; i + 4 <= n; i += kMlpBlock * 4) *reinterpret_cast<float4*>(d + i) = ld4(g + i, true);
    for (i = (n & ~3) + threadIdx.x; i < n; i += kMlpBlock) d[i] = g[i];
  } else {
    for (i = threadIdx.x; i < n; i += kMlpBlock) d[i] = g[i];
  }
}

// Every sum runs over its terms in order, one FMA a term, starting from the bias.
__global__ void __launch_bounds__(kMlpBlock) k_mlp_forward(const __grid_constant__ MlpArgs a) {
  extern __shared__ float4 smem4[];
  float* sp = reinterpret_cast<float*>(smem4);
  const int F = a.F;
  const int np = static_cast<int>(mlp_n_params(F));
  float* xt = sp + ((np + 3) & ~3);  // [F][kLd]: inputs by feature
  float* ht = xt + F * kLd;          // [kH][kLd]: activations by unit
  stage_floats(sp, a.p, np);
  const float* W1 = sp;
  const float* b1 = W1 + F * kH;
  const float* W2 = b1 + kH;
  const float* b2 = W2 + kH * kH;
  const float* w3 = b2 + kH;
  const int64_t i0 = static_cast<int64_t>(blockIdx.x) * kTile;
  const int n = static_cast<int>(a.B - i0 < kTile ? a.B - i0 : kTile);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int s = warp; s < kTile; s += kMlpBlock / 32)
    for (int f = lane; f < F; f += 32) xt[f * kLd + s] = s < n ? (a.x[(i0 + s) * F + f] - a.mu[f]) / a.sigma[f] : 0.0f;
  __syncthreads();
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;  // units 4 tx ..., samples 4 ty ...
  const bool vec = aligned16(a.act);
  float z[4][4];
  // z = bias + (tile by input) (input by unit), kept as sample by unit
  auto product = [&](const float* in, const float* W, const float* bias, int K) {
    const float4 b = lds4(bias + 4 * tx);
#pragma unroll
    for (int i = 0; i < 4; ++i) { z[i][0] = b.x; z[i][1] = b.y; z[i][2] = b.z; z[i][3] = b.w; }
#pragma unroll 4
    for (int k = 0; k < K; ++k) {
      const float4 x4 = lds4(in + k * kLd + 4 * ty), w4 = lds4(W + k * kH + 4 * tx);
      const float x[4] = {x4.x, x4.y, x4.z, x4.w}, w[4] = {w4.x, w4.y, w4.z, w4.w};
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) z[i][j] = fmaf(x[i], w[j], z[i][j]);
    }
  };
  auto store_act = [&](int off) {
    if (a.act == nullptr) return;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      if (4 * ty + i >= n) continue;
      float* o = a.act + (i0 + 4 * ty + i) * 2 * kH + off + 4 * tx;
      if (vec) {
        *reinterpret_cast<float4*>(o) = make_float4(z[i][0], z[i][1], z[i][2], z[i][3]);
      } else {
#pragma unroll
        for (int j = 0; j < 4; ++j) o[j] = z[i][j];
      }
    }
  };
  auto store_relu = [&]() {  // by unit
#pragma unroll
    for (int j = 0; j < 4; ++j)
      *reinterpret_cast<float4*>(ht + (4 * tx + j) * kLd + 4 * ty) =
          make_float4(fmaxf(z[0][j], 0.0f), fmaxf(z[1][j], 0.0f), fmaxf(z[2][j], 0.0f), fmaxf(z[3][j], 0.0f));
  };
  product(xt, W1, b1, F);
  store_act(0);
  store_relu();
  __syncthreads();
  product(ht, W2, b2, kH);
  store_act(kH);
  __syncthreads();
  store_relu();
  __syncthreads();
  if (threadIdx.x < n) {
    float y = w3[kH];
#pragma unroll 16
    for (int k = 0; k < kH; ++k) y = fmaf(ht[k * kLd + threadIdx.x], w3[k], y);
    a.y[i0 + threadIdx.x] = y;
  }
}

// Adds v[0..3] to g[0..3]; vec: g is 16-byte aligned (one reduction of 4 floats).
__device__ __forceinline__ void grad_add4(float* g, const float (&v)[4], bool vec) {
  if (vec) {
    asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(g), "f"(v[0]), "f"(v[1]), "f"(v[2]), "f"(v[3])
                 : "memory");
  } else {
#pragma unroll
    for (int j = 0; j < 4; ++j) atomicAdd(g + j, v[j]);
  }
}

// Backward: dy = 2 (y - t) / B, dz2 = dy w3 (z2 > 0), dz1 = (W2 dz2)(z1 > 0),
// the loss and every gradient.  A CTA takes tiles of 16 * MS samples; its
// threads keep 4 x 4 blocks of both weight gradients over all of its tiles
// and add them to one of the copies of the gradient at its end, four floats at
// a time: with one copy for all CTAs the sums would round once per CTA.  The per-sample deltas stay in shared memory.
template <int MS>
constexpr int mlp_backward_floats() { return 16 * MS * (4 * kH + 1) + kH * kLd + kH; }

template <int MS>
__global__ void __launch_bounds__(kMlpBlock, 2) k_mlp_backward(const __grid_constant__ MlpArgs a) {
  constexpr int TS = 16 * MS;
  static_assert(4 * TS >= 3 * 16, "the tile's buffers hold the vectors' partial sums");
  extern __shared__ float4 smem4[];
  float* xh = reinterpret_cast<float*>(smem4);  // [TS][kH], columns past F zero
  float* h1 = xh + TS * kH;                     // [TS][kH]
  float* d1 = h1 + TS * kH;                     // [TS][kH]
  float* d2 = d1 + TS * kH;                     // [TS][kH]
  float* W2t = d2 + TS * kH;                    // [k][kLd]: W2 by output unit
  float* w3 = W2t + kH * kLd;                   // [kH]
  float* dy = w3 + kH;                          // [TS]
  const int F = a.F;
  const float* W2 = a.p + F * kH + kH;
  for (int e = threadIdx.x; e < kH * kH; e += kMlpBlock) W2t[(e & (kH - 1)) * kLd + e / kH] = W2[e];
  if (threadIdx.x < kH) w3[threadIdx.x] = W2[kH * kH + kH + threadIdx.x];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  const bool vec = aligned16(a.act);
  float g1[4][4] = {}, g2[4][4] = {};             // inputs (units) 4 ty ..., units 4 tx ...
  float gb1[4] = {}, gb2[4] = {}, gw3[4] = {};  // units 4 tx ...
  float gb3 = 0.0f, loss = 0.0f;
  const int64_t n_tiles = (a.B + TS - 1) / TS;
  for (int64_t tile = blockIdx.x; tile < n_tiles; tile += gridDim.x) {
    const int64_t i0 = tile * TS;
    const int n = static_cast<int>(a.B - i0 < TS ? a.B - i0 : TS);
    if (threadIdx.x < TS) {
      float v = 0.0f;
      if (threadIdx.x < n) {
        const float d = a.y[i0 + threadIdx.x] - a.t[i0 + threadIdx.x];
        loss += d * d / a.B;
        v = 2.0f * d / a.B;
      }
      dy[threadIdx.x] = v;
      gb3 += v;
    }
    for (int s = warp; s < TS; s += kMlpBlock / 32)
#pragma unroll
      for (int f = lane; f < kH; f += 32)
        xh[s * kH + f] = s < n && f < F ? (a.x[(i0 + s) * F + f] - a.mu[f]) / a.sigma[f] : 0.0f;
    __syncthreads();
#pragma unroll
    for (int q = 0; q < MS; ++q) {
      const int s = ty + 16 * q;
      float4 z1 = make_float4(0, 0, 0, 0), z2 = z1;
      if (s < n) {
        const float* o = a.act + (i0 + s) * 2 * kH + 4 * tx;
        z1 = ld4(o, vec);
        z2 = ld4(o + kH, vec);
      }
      const float v = dy[s];
      const float4 w = lds4(w3 + 4 * tx);
      const float z[4] = {z2.x, z2.y, z2.z, z2.w}, wv[4] = {w.x, w.y, w.z, w.w};
      float d[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        d[j] = z[j] > 0.0f ? v * wv[j] : 0.0f;
        gb2[j] += d[j];
        gw3[j] = fmaf(fmaxf(z[j], 0.0f), v, gw3[j]);
      }
      *reinterpret_cast<float4*>(d2 + s * kH + 4 * tx) = make_float4(d[0], d[1], d[2], d[3]);
      *reinterpret_cast<float4*>(h1 + s * kH + 4 * tx) =
          make_float4(fmaxf(z1.x, 0.0f), fmaxf(z1.y, 0.0f), fmaxf(z1.z, 0.0f), fmaxf(z1.w, 0.0f));
    }
    __syncthreads();
    // dz1: samples MS * ty ..., units 4 tx ...
    {
      float z[MS][4] = {};
#pragma unroll 2
      for (int k = 0; k < kH; k += 4) {
        float4 d[MS];
#pragma unroll
        for (int i = 0; i < MS; ++i) d[i] = lds4(d2 + (MS * ty + i) * kH + k);
#pragma unroll
        for (int kk = 0; kk < 4; ++kk) {
          const float4 w4 = lds4(W2t + (k + kk) * kLd + 4 * tx);
#pragma unroll
          for (int i = 0; i < MS; ++i) {
            const float dv = kk == 0 ? d[i].x : kk == 1 ? d[i].y : kk == 2 ? d[i].z : d[i].w;
            z[i][0] = fmaf(w4.x, dv, z[i][0]);
            z[i][1] = fmaf(w4.y, dv, z[i][1]);
            z[i][2] = fmaf(w4.z, dv, z[i][2]);
            z[i][3] = fmaf(w4.w, dv, z[i][3]);
          }
        }
      }
#pragma unroll
      for (int i = 0; i < MS; ++i) {
        const int at = (MS * ty + i) * kH + 4 * tx;
        const float4 h = lds4(h1 + at);
        const float hv[4] = {h.x, h.y, h.z, h.w};
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          z[i][j] = hv[j] > 0.0f ? z[i][j] : 0.0f;
          gb1[j] += z[i][j];
        }
        *reinterpret_cast<float4*>(d1 + at) = make_float4(z[i][0], z[i][1], z[i][2], z[i][3]);
      }
    }
    __syncthreads();
    // Weight gradients of the tile: (rows by input)^T (rows by unit).
    auto outer = [&](const float* in, const float* d, float (&g)[4][4]) {
#pragma unroll 1
      for (int s0 = 0; s0 < TS; s0 += 16) {  // sums of 16 samples first: shorter rounding chains
        float t[4][4] = {};
#pragma unroll 4
        for (int s = s0; s < s0 + 16; ++s) {
          const float4 x4 = lds4(in + s * kH + 4 * ty), d4 = lds4(d + s * kH + 4 * tx);
          const float x[4] = {x4.x, x4.y, x4.z, x4.w}, dv[4] = {d4.x, d4.y, d4.z, d4.w};
#pragma unroll
          for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) t[i][j] = fmaf(x[i], dv[j], t[i][j]);
        }
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
          for (int j = 0; j < 4; ++j) g[i][j] += t[i][j];
      }
    };
    if (4 * ty < F) outer(xh, d1, g1);
    outer(h1, d2, g2);
    __syncthreads();  // the tile's buffers are free again
  }
  const int64_t copy = static_cast<int64_t>(blockIdx.x % a.copies) * a.stride;
  float* oW1 = a.grad + copy;
  float* ob1 = oW1 + F * kH;
  float* oW2 = ob1 + kH;
  float* ob2 = oW2 + kH * kH;  // then w3, b3
  const bool gvec = aligned16(oW1);
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    if (4 * ty + i < F) grad_add4(oW1 + (4 * ty + i) * kH + 4 * tx, g1[i], gvec);
    grad_add4(oW2 + (4 * ty + i) * kH + 4 * tx, g2[i], gvec);
  }
  // the vectors: partial sums of the 16 thread rows, then one add per unit
  float* red = xh;  // [3][16][kH], over the tile's buffers
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    red[ty * kH + 4 * tx + j] = gb1[j];
    red[(16 + ty) * kH + 4 * tx + j] = gb2[j];
    red[(32 + ty) * kH + 4 * tx + j] = gw3[j];
  }
  __syncthreads();
  if (threadIdx.x < 3 * kH) {
    const int which = threadIdx.x / kH, j = threadIdx.x % kH;
    float v = 0.0f;
#pragma unroll
    for (int r = 0; r < 16; ++r) v += red[(16 * which + r) * kH + j];
    atomicAdd((which == 0 ? ob1 : which == 1 ? ob2 : ob2 + kH) + j, v);
  }
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    gb3 += __shfl_xor_sync(0xffffffffu, gb3, off);
    loss += __shfl_xor_sync(0xffffffffu, loss, off);
  }
  if (lane == 0 && warp * 32 < TS) {
    atomicAdd(ob2 + 2 * kH, gb3);
    atomicAdd(a.loss + copy, loss);
  }
  pdl_launch_dependents();
}

// Gradient and loss from their copies, each rounded once.
__global__ void k_mlp_sum(const float* part, int copies, int64_t stride, int np, float* grad, float* loss) {
  pdl_wait();  // launched early behind the backward kernel
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i > np) return;
  double v = 0.0;
  for (int c = 0; c < copies; ++c) v += part[c * stride + i];
  if (i < np) grad[i] = static_cast<float>(v);
  else *loss = static_cast<float>(v);
}

__global__ void k_mlp_adam(float* p, const float* g, float* m, float* v, int64_t n, float lr, float b1, float b2,
                           float eps, float c1, float c2) {
  for (int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; i < n;
       i += static_cast<int64_t>(gridDim.x) * blockDim.x) {
    const float gi = g[i];
    const float mi = b1 * m[i] + (1.0f - b1) * gi;
    const float vi = b2 * v[i] + (1.0f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    p[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
  }
}

pv_status mlp_forward(cudaStream_t s, int* launches, const float* params, const float* x, const float* mu,
                      const float* sigma, int B, int F, float* y, float* act) {
  if (B < 0 || F < 1 || F > kMaxF || !params || !x || !mu || !sigma || (B > 0 && !y)) return PV_ERR_INVALID_ARG;
  if (B == 0) return PV_OK;
  MlpArgs a{};
  a.p = params; a.x = x; a.mu = mu; a.sigma = sigma; a.y = y; a.act = act; a.B = B; a.F = F;
  const size_t smem = (static_cast<size_t>((mlp_n_params(F) + 3) & ~3ll) + static_cast<size_t>(F + kH) * kLd) * sizeof(float);
  if (cudaFuncSetAttribute(k_mlp_forward, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem)) != cudaSuccess)
    return PV_ERR_CUDA;
  k_mlp_forward<<<(B - 1) / kTile + 1, kMlpBlock, smem, s>>>(a);
  ++*launches;
  return cudaGetLastError() == cudaSuccess ? PV_OK : PV_ERR_CUDA;
}

template <int MS>
static cudaError_t launch_backward(cudaStream_t s, const MlpArgs& a, int max_ctas) {
  const size_t smem = mlp_backward_floats<MS>() * sizeof(float);
  const cudaError_t e = cudaFuncSetAttribute(k_mlp_backward<MS>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             static_cast<int>(smem));
  if (e != cudaSuccess) return e;
  k_mlp_backward<MS><<<std::min((a.B - 1) / (16 * MS) + 1, max_ctas), kMlpBlock, smem, s>>>(a);
  return cudaGetLastError();
}

pv_status mlp_backward(cudaStream_t s, int* launches, const float* params, const float* x, const float* mu,
                       const float* sigma, const float* act, const float* y, const float* t, int B, int F,
                       float* dz, float* grad, float* loss) {
  if (B < 1 || F < 1 || F > kMaxF || !params || !x || !mu || !sigma || !act || !y || !t || !dz || !grad || !loss)
    return PV_ERR_INVALID_ARG;
  MlpArgs a{};
  a.p = params; a.x = x; a.mu = mu; a.sigma = sigma; a.y = const_cast<float*>(y); a.act = const_cast<float*>(act);
  a.t = t; a.grad = grad; a.loss = loss; a.B = B; a.F = F;
  // Up to 16 copies of the gradient and the loss in dz (B x (2H + 1) floats), else the outputs themselves.
  const int np = static_cast<int>(mlp_n_params(F));
  a.stride = (np + 1 + 3) & ~3;
  const int64_t room = static_cast<int64_t>(B) * (2 * kH + 1) / a.stride;
  const int copies = static_cast<int>(std::min<int64_t>(16, room));
  a.copies = std::max(1, copies);
  if (copies > 0) {
    a.grad = dz;
    a.loss = dz + np;
    if (cudaMemsetAsync(dz, 0, static_cast<size_t>(copies) * a.stride * sizeof(float), s) != cudaSuccess) return PV_ERR_CUDA;
  } else {
    if (cudaMemsetAsync(grad, 0, static_cast<size_t>(np) * sizeof(float), s) != cudaSuccess) return PV_ERR_CUDA;
    if (cudaMemsetAsync(loss, 0, sizeof(float), s) != cudaSuccess) return PV_ERR_CUDA;
  }
  int dev = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
    return PV_ERR_CUDA;
  // Two CTAs an SM.  The tile (32 to 80 samples) that leaves the busiest CTA the fewest sample slots:
  // its last tile may be mostly empty, and small batches want small tiles on many SMs.
  const int ctas = 2 * sms;
  int best = 5;
  int64_t cost = INT64_MAX;
  for (int ms = 5; ms >= 2; --ms) {
    const int64_t tiles = (B - 1) / (16 * ms) + 1;
    const int64_t c = ((tiles - 1) / ctas + 1) * ms;
    if (c < cost) { cost = c; best = ms; }
  }
  const cudaError_t e = best == 5   ? launch_backward<5>(s, a, ctas)
                        : best == 4 ? launch_backward<4>(s, a, ctas)
                        : best == 3 ? launch_backward<3>(s, a, ctas)
                                    : launch_backward<2>(s, a, ctas);
  if (e != cudaSuccess) return PV_ERR_CUDA;
  ++*launches;
  if (copies > 0) {
    if (pdl_launch(k_mlp_sum, dim3(np / 256 + 1), dim3(256), 0, s, static_cast<const float*>(dz), copies, a.stride, np,
                   grad, loss) != cudaSuccess)
      return PV_ERR_CUDA;
    ++*launches;
  }
  return PV_OK;
}

pv_status mlp_adam(cudaStream_t s, int* launches, float* p, const float* g, float* m, float* v, int64_t n, float lr,
                   float b1, float b2, float eps, int step) {
  if (!p || !g || !m || !v || n < 0 || step < 1 || !(b1 >= 0 && b1 < 1) || !(b2 >= 0 && b2 < 1)) return PV_ERR_INVALID_ARG;
  if (n == 0) return PV_OK;
  const float c1 = 1.0f - powf(b1, static_cast<float>(step));
  const float c2 = 1.0f - powf(b2, static_cast<float>(step));
  const int grid = static_cast<int>(std::min<int64_t>(1024, (n + 255) / 256));
  k_mlp_adam<<<grid, 256, 0, s>>>(p, g, m, v, n, lr, b1, b2, eps, c1, c2);
  ++*launches;
  return cudaGetLastError() == cudaSuccess ? PV_OK : PV_ERR_CUDA;
}

}  // namespace pv
