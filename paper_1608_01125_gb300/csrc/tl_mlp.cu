// tl_mlp.cu -- the surrogate network: 24 -> 128 -> 128 -> 128 -> 2, exact
// GELU between layers, BF16 weights and activations with FP32 accumulation.
//
// Every product runs on the tensor cores (tcgen05.mma, accumulators in tensor
// memory): each layer is a 128 x N x K tile product issued by one thread; its FP32
// result is read back row per thread (tcgen05.ld), biased, activated and written as
// the next layer's BF16 operand.  Inference: four groups of 128 threads per block,
// each with a 128-row tile of its own (k_mlp_forward).  Training: forward, input
// gradients and weight gradients of a tile in one kernel, nothing but the weight
// gradients leaving the SM (k_mlp_grad); the optimiser on the CUDA cores.
//
// Outputs per row: mu and s (log variance) of a Gaussian over
// y = log1p(sum of w_i w_j of a node pair).  Loss 0.5 (s + (y - mu)^2 e^-s),
// s clamped to +-12, mean over the batch.
#include <cuda_bf16.h>
#include <stddef.h>
#include <string.h>

#include <mutex>

#include "tl_sur.h"
#include "tl_tc.cuh"
#include "trilens.h"

namespace tl {

constexpr int kIn = 24, kInP = 32, kH = 128, kOutP = 16;
// flat FP32 parameter vector: W1 (128x24), b1, W2 (128x128), b2, W3, b3, W4 (2x128), b4
constexpr int kOffW1 = 0, kOffB1 = kOffW1 + kH * kIn, kOffW2 = kOffB1 + kH,
              kOffB2 = kOffW2 + kH * kH, kOffW3 = kOffB2 + kH, kOffB3 = kOffW3 + kH * kH,
              kOffW4 = kOffB3 + kH, kOffB4 = kOffW4 + 2 * kH, kParams = kOffB4 + 2;
static_assert(kParams == TRILENS_MLP_PARAMS, "parameter count");
constexpr float kSClamp = 12.0f;
constexpr int kGroups = 4, kThreads = 128 * kGroups;

__device__ __forceinline__ float gelu(float x) {
  return 0.5f * x * (1.0f + erff(x * 0.70710678118654752f));
}
__device__ __forceinline__ float gelu_grad(float x) {
  return 0.5f * (1.0f + erff(x * 0.70710678118654752f)) +
         x * 0.39894228040143268f * __expf(-0.5f * x * x);
}

template <class T>
__device__ __forceinline__ T *align1k(unsigned char *p) {
  return reinterpret_cast<T *>((reinterpret_cast<uintptr_t>(p) + 1023) & ~(uintptr_t)1023);
}

// ---------------------------------------------------------------- operand tiles

// write 8 consecutive values of row r (columns c..c+7) into a core tile
__device__ __forceinline__ void put8(__nv_bfloat16 *tile, int r, int c, int K, const float *v) {
  __align__(16) __nv_bfloat162 h[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) h[j] = __floats2bfloat162_rn(v[2 * j], v[2 * j + 1]);
  *reinterpret_cast<uint4 *>(tile + core_idx(r, c, K)) = *reinterpret_cast<const uint4 *>(h);
}

// FP32 weights [R][C] -> BF16 core tile of R x K (columns C.. and rows rows.. zero).
// Every block converts its own copy from the FP32 parameters (146 KB, in L2), so no
// packed copy of the weights has to be kept or made first.
__device__ __forceinline__ void load_w(__nv_bfloat16 *dst, const float *src, int R, int K, int rows,
                                       int C) {
  for (int idx = threadIdx.x; idx < R * K / 8; idx += kThreads) {
    const int r = idx / (K / 8), k = (idx - r * (K / 8)) * 8;
    float v[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) v[j] = r < rows && k + j < C ? __ldg(src + r * C + k + j) : 0.0f;
    put8(dst, r, k, K, v);
  }
}

// transposed: dst(n, k) = src[k][n], src [rows][N] row-major, rows past `rows` zero
__device__ __forceinline__ void load_wt(__nv_bfloat16 *dst, const float *src, int N, int K,
                                        int rows) {
  for (int idx = threadIdx.x; idx < N * K / 8; idx += kThreads) {
    const int n = idx % N, k = (idx / N) * 8;  // neighbouring threads: neighbouring n
    float v[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) v[j] = k + j < rows ? __ldg(src + (k + j) * N + n) : 0.0f;
    put8(dst, n, k, K, v);
  }
}

// (operand tiles in shared memory start on 128-byte boundaries: descriptors and 16-byte
// stores need 16)
struct Weights {  // the forward products' B operands and the biases
  alignas(128) __nv_bfloat16 W1[kH * kInP];
  alignas(128) __nv_bfloat16 W2[kH * kH];
  alignas(128) __nv_bfloat16 W3[kH * kH];
  alignas(128) __nv_bfloat16 W4[kOutP * kH];
  float b[3][kH];
  float b4[2];
  float norm[2 * kIn];  // feature mean, 1 / std
};

__device__ __forceinline__ void load_weights(Weights &S, const float *prm, const float *norm) {
  load_w(S.W1, prm + kOffW1, kH, kInP, kH, kIn);
  load_w(S.W2, prm + kOffW2, kH, kH, kH, kH);
  load_w(S.W3, prm + kOffW3, kH, kH, kH, kH);
  load_w(S.W4, prm + kOffW4, kOutP, kH, 2, kH);
  for (int j = threadIdx.x; j < kH; j += kThreads) {
    S.b[0][j] = prm[kOffB1 + j];
    S.b[1][j] = prm[kOffB2 + j];
    S.b[2][j] = prm[kOffB3 + j];
  }
  for (int j = threadIdx.x; j < 2 * kIn; j += kThreads) S.norm[j] = norm[j];
  if (threadIdx.x < 2) S.b4[threadIdx.x] = prm[kOffB4 + threadIdx.x];
}

// the normalised features c..c+7 of a row (zero past the features or the batch)
__device__ __forceinline__ void features8(const float *x, int64_t row, bool valid,
                                          const float *norm, int c, float *v) {
#pragma unroll
  for (int j = 0; j < 8; ++j)
    v[j] = valid && c + j < kIn ? (x[row * kIn + c + j] - norm[c + j]) * norm[kIn + c + j] : 0.0f;
}

__device__ __forceinline__ void set_error(int *err) {
  *(volatile int *)err = 1;
  __threadfence_system();
}

// ---------------------------------------------------------------- forward

struct FwdSmem {
  Weights w;
  alignas(128) __nv_bfloat16 A[kGroups][128 * kH];
  uint64_t mbar[kGroups];
  uint32_t tmem;
};

__device__ __forceinline__ void group_sync(int g) {
  asm volatile("bar.sync %0, 128;" ::"r"(1 + g) : "memory");
}

// One layer of a group's tile: product, then a bounded wait for it.
__device__ __forceinline__ bool group_mma(FwdSmem &S, int g, uint32_t d, const void *B, int K, int N,
                                          uint32_t &phase, long long spin) {
  fence_async_smem();
  tc_fence_before();
  group_sync(g);
  tc_fence_after();
  if ((threadIdx.x & 127) == 0) {
    gemm_tile(d, S.A[g], B, K, N, false);
    mma_commit(&S.mbar[g]);
  }
  const bool ok = mbar_wait(&S.mbar[g], phase, spin);
  phase ^= 1u;
  tc_fence_after();
  return ok;
}

// Inference over M rows of raw features x [M][24] -> out [M][2].  What bounds it is the
// GELU on the CUDA cores (384 erff per row against 72 kFLOP of products); one group of
// 128 threads per SM left its schedulers idle between dependent instructions and during
// its own products, so a block runs four groups, each with its own rows, accumulator
// columns and barrier, around one copy of the weights.  A call for 200,003 rows: 423 us with
// one group and allocations on every call (197 us of it the kernel), 137 us now.
__global__ void __launch_bounds__(kThreads, 1)
    k_mlp_forward(const float *__restrict__ prm, const float *__restrict__ norm,
                  const float *__restrict__ x, int64_t M, float *out, int *err, long long spin) {
  extern __shared__ unsigned char smem_raw[];
  FwdSmem &S = *align1k<FwdSmem>(smem_raw);
  const int tid = threadIdx.x, g = tid >> 7, gt = tid & 127, warp = tid >> 5;
  load_weights(S.w, prm, norm);
  if (tid < kGroups) mbar_init(&S.mbar[tid], 1);
  if (warp == 0) {
    tmem_alloc(&S.tmem, 512);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = S.tmem + (uint32_t)(g * kH);
  const uint32_t trow = tmem + ((uint32_t)((warp & 3) * 32) << 16);
  uint32_t phase = 0;
  bool ok = true;
  const int64_t ntiles = (M + 127) / 128;
  for (int64_t tile = blockIdx.x + (int64_t)gridDim.x * g; tile < ntiles;
       tile += (int64_t)gridDim.x * kGroups) {
    const int64_t row = tile * 128 + gt;
    const bool valid = row < M;
#pragma unroll
    for (int c = 0; c < kInP; c += 8) {
      float v[8];
      features8(x, row, valid, S.w.norm, c, v);
      put8(S.A[g], gt, c, kInP, v);
    }
    ok = group_mma(S, g, tmem, S.w.W1, kInP, kH, phase, spin) && ok;
#pragma unroll 1
    for (int l = 0; l < 3; ++l) {
      // epilogue of layer l + 1: bias, GELU -> next operand
      const float *bias = S.w.b[l];
#pragma unroll 1
      for (int c = 0; c < kH; c += 16) {
        uint32_t r[16];
        TL_TMEM_LD_X16(trow + (uint32_t)c, r);
        tmem_wait_ld();
        float h[16];
#pragma unroll
        for (int j = 0; j < 16; ++j) h[j] = gelu(__uint_as_float(r[j]) + bias[c + j]);
        put8(S.A[g], gt, c, kH, h);
        put8(S.A[g], gt, c + 8, kH, h + 8);
      }
      ok = group_mma(S, g, tmem, l == 0 ? S.w.W2 : (l == 1 ? S.w.W3 : S.w.W4), kH,
                     l < 2 ? kH : kOutP, phase, spin) && ok;
    }
    uint32_t r[16];
    TL_TMEM_LD_X16(trow, r);
    tmem_wait_ld();
    if (valid) {
      out[2 * row] = __uint_as_float(r[0]) + S.w.b4[0];
      out[2 * row + 1] = __uint_as_float(r[1]) + S.w.b4[1];
    }
    tc_fence_before();
    group_sync(g);  // the accumulator and the operand are read before the next tile
    tc_fence_after();
  }
  if (!ok) set_error(err);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 0) tmem_dealloc(S.tmem, 512);
}

// ---------------------------------------------------------------- gradients

struct GradSmem {
  Weights w;
  alignas(128) __nv_bfloat16 W2T[kH * kH];
  alignas(128) __nv_bfloat16 W3T[kH * kH];
  alignas(128) __nv_bfloat16 W4T[kH * kOutP];
  alignas(128) __nv_bfloat16 T0[128 * kH];
  alignas(128) __nv_bfloat16 T1[128 * kH];
  alignas(128) __nv_bfloat16 O[128 * kOutP];   // dout, row-major
  alignas(128) __nv_bfloat16 OT[kOutP * 128];  // dout transposed
  float loss[4];
  uint64_t mbar;
  uint32_t tmem;
};

// store (first) or add a value of the block's slice of the gradients
__device__ __forceinline__ void part_put(float *p, float v, bool first) {
  *p = first ? v : *p + v;
}

// Loss and gradients of the mean loss.  A block takes 128-row tiles; for each it runs the
// forward pass (pre-activations of the three hidden layers stay in tensor memory), the
// loss, the input gradients and the weight gradients, 512 threads on the tile (group g
// reads accumulator columns 32 g..), and writes its sums to its own slice of `part`;
// k_mlp_wsum adds the slices in block order, so the gradient is reproducible bit for
// bit.  The input gradients are products with the transposed weights.  The weight
// gradients are products over the batch: dW[o][i] = sum_r G[r][o] H[r][i], A = G^T and
// B = H^T staged as K-major tiles with the rows as K (layer 4 transposed: A = H3^T,
// B = dout^T).  H is GELU of the BF16 pre-activation, G the BF16 upstream gradient.
// What bounds it is the chain of ten products and their epilogues, a few us each; kernels
// of their own for forward, input gradients and four weight gradients, exchanging
// activations through memory and staging operands with 2-byte strided loads, took 518 us
// for 8192 rows, this and the sum 81 us.
//
// Loss kind 0: Gaussian NLL of y with (mu, s).  Kind 1 (the surrogate's): y is the linear
// label Y, B = st_scale * st[row] the baseline, lam = (B + 1) e^mu the predicted mean;
// loss (lam - Y ln lam)/(B + 1) + 0.5 (s + r^2 e^-s), r = log1p(Y) - log1p(lam) with lam
// held fixed in r.
__global__ void __launch_bounds__(kThreads, 1)
    k_mlp_grad(const float *__restrict__ prm, const float *__restrict__ norm,
               const float *__restrict__ x, const float *__restrict__ y, int64_t M, float *part,
               float *part_loss, float inv_b, int *err, long long spin, int kind,
               const float *__restrict__ st, float st_scale) {
  extern __shared__ unsigned char smem_raw[];
  GradSmem &S = *align1k<GradSmem>(smem_raw);
  const int tid = threadIdx.x, g = tid >> 7, gt = tid & 127, warp = tid >> 5;
  load_weights(S.w, prm, norm);
  load_wt(S.W2T, prm + kOffW2, kH, kH, kH);
  load_wt(S.W3T, prm + kOffW3, kH, kH, kH);
  load_wt(S.W4T, prm + kOffW4, kH, kOutP, 2);
  if (tid == 0) mbar_init(&S.mbar, 1);
  if (warp == 0) {
    tmem_alloc(&S.tmem, 512);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tm = S.tmem;
  const uint32_t lanes = (uint32_t)((warp & 3) * 32) << 16;
  const uint32_t zc[3] = {tm, tm + 128u, tm + 256u}, dc = tm + 384u, ac = zc[2];
  const int c0 = 32 * g;  // this thread's columns
  uint32_t phase = 0;
  bool ok = true;
  float *P = part + (size_t)blockIdx.x * kParams;
  float lsum = 0.0f;
  bool first = true;

  // operands written -> visible to the tensor cores, accumulators read
  auto ready = [&]() {
    fence_async_smem();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
  };
  auto wait = [&]() {
    ok = mbar_wait(&S.mbar, phase, spin) && ok;
    phase ^= 1u;
    tc_fence_after();
  };
  // pre-activations of layer l + 1 as BF16 pairs, this thread's 32 columns
  auto load_z = [&](int l, uint32_t *zb) {
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      uint32_t r[16];
      TL_TMEM_LD_X16(zc[l] + lanes + (uint32_t)(c0 + 16 * h), r);
      tmem_wait_ld();
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const int c = c0 + 16 * h + 2 * j;
        const __nv_bfloat162 v = __floats2bfloat162_rn(__uint_as_float(r[2 * j]) + S.w.b[l][c],
                                                       __uint_as_float(r[2 * j + 1]) + S.w.b[l][c + 1]);
        zb[8 * h + j] = *reinterpret_cast<const uint32_t *>(&v);
      }
    }
  };
  auto unpack = [](uint32_t v) {
    return __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&v));
  };
  // GELU of BF16 pre-activations, transposed into a tile (row = input, K = batch row)
  auto stage_ht = [&](__nv_bfloat16 *T, const uint32_t *zb, bool valid) {
#pragma unroll
    for (int j = 0; j < 16; ++j) {
      const float2 z = unpack(zb[j]);
      T[core_idx(c0 + 2 * j, gt, 128)] = __float2bfloat16(valid ? gelu(z.x) : 0.0f);
      T[core_idx(c0 + 2 * j + 1, gt, 128)] = __float2bfloat16(valid ? gelu(z.y) : 0.0f);
    }
  };
  // G = (product in dc) gelu'(Z), as BF16 pairs
  auto upstream = [&](const uint32_t *zb, bool valid, uint32_t *gp) {
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      uint32_t r[16];
      TL_TMEM_LD_X16(dc + lanes + (uint32_t)(c0 + 16 * h), r);
      tmem_wait_ld();
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const float2 z = unpack(zb[8 * h + j]);
        const float a = valid ? __uint_as_float(r[2 * j]) * gelu_grad(z.x) : 0.0f;
        const float b = valid ? __uint_as_float(r[2 * j + 1]) * gelu_grad(z.y) : 0.0f;
        const __nv_bfloat162 v = __floats2bfloat162_rn(a, b);
        gp[8 * h + j] = *reinterpret_cast<const uint32_t *>(&v);
      }
    }
  };
  auto put_rows = [&](__nv_bfloat16 *T, const uint32_t *gp) {  // row-major operand
#pragma unroll
    for (int q = 0; q < 4; ++q)
      *reinterpret_cast<uint4 *>(T + core_idx(gt, c0 + 8 * q, kH)) =
          make_uint4(gp[4 * q], gp[4 * q + 1], gp[4 * q + 2], gp[4 * q + 3]);
  };
  auto stage_gt = [&](__nv_bfloat16 *T, const uint32_t *gp) {  // transposed
#pragma unroll
    for (int j = 0; j < 16; ++j) {
      const __nv_bfloat162 v = *reinterpret_cast<const __nv_bfloat162 *>(&gp[j]);
      T[core_idx(c0 + 2 * j, gt, 128)] = v.x;
      T[core_idx(c0 + 2 * j + 1, gt, 128)] = v.y;
    }
  };
  // bias gradient of output gt from the staged G^T (one group), rows in order
  auto bias_grad = [&](const __nv_bfloat16 *T, float *db) {
    if (g != 3) return;
    float a = 0.0f;
    for (int k = 0; k < 128; k += 8) {
      const uint4 v = *reinterpret_cast<const uint4 *>(T + core_idx(gt, k, 128));
      const uint32_t u[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const float2 f = unpack(u[j]);
        a += f.x;
        a += f.y;
      }
    }
    part_put(db + gt, a, first);
  };
  // accumulator rows -> the slice: output gt, columns c0.. (n columns in all)
  auto write_w = [&](float *dW, int n) {
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int c = c0 + 16 * h;
      uint32_t r[16];
      if (c0 < n) {  // (uniform over a group)
        TL_TMEM_LD_X16(ac + lanes + (uint32_t)c, r);
        tmem_wait_ld();
#pragma unroll
        for (int j = 0; j < 16; ++j)
          if (c + j < n) part_put(dW + gt * n + c + j, __uint_as_float(r[j]), first);
      }
    }
  };

  const int64_t ntiles = (M + 127) / 128;
  for (int64_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
    const int64_t row = tile * 128 + gt;
    const bool valid = row < M;
    // ---- forward
    {
      float v[8];
      features8(x, row, valid, S.w.norm, 8 * g, v);
      put8(S.T0, gt, 8 * g, kInP, v);
    }
    ready();
    if (tid == 0) {
      gemm_tile(zc[0], S.T0, S.w.W1, kInP, kH, false);
      mma_commit(&S.mbar);
    }
    wait();
#pragma unroll 1
    for (int l = 0; l < 3; ++l) {
      __nv_bfloat16 *T = l == 1 ? S.T0 : S.T1;
#pragma unroll 1
      for (int c = c0; c < c0 + 32; c += 16) {
        uint32_t r[16];
        TL_TMEM_LD_X16(zc[l] + lanes + (uint32_t)c, r);
        tmem_wait_ld();
        float h[16];
#pragma unroll
        for (int j = 0; j < 16; ++j) h[j] = gelu(__uint_as_float(r[j]) + S.w.b[l][c + j]);
        put8(T, gt, c, kH, h);
        put8(T, gt, c + 8, kH, h + 8);
      }
      ready();
      if (tid == 0) {
        gemm_tile(l == 0 ? zc[1] : (l == 1 ? zc[2] : dc), T,
                  l == 0 ? S.w.W2 : (l == 1 ? S.w.W3 : S.w.W4), kH, l < 2 ? kH : kOutP, false);
        mma_commit(&S.mbar);
      }
      wait();
    }
    // ---- loss and its gradient
    uint32_t zb[16], gp[16];
    load_z(2, zb);
    if (g == 0) {
      uint32_t r[16];
      TL_TMEM_LD_X16(dc + lanes, r);
      tmem_wait_ld();
      const float o0 = __uint_as_float(r[0]) + S.w.b4[0], o1 = __uint_as_float(r[1]) + S.w.b4[1];
      float d[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
      if (valid) {
        const float s = fminf(fmaxf(o1, -kSClamp), kSClamp), e = __expf(-s);
        const bool in = o1 > -kSClamp && o1 < kSClamp;
        if (kind == 0) {
          const float res = y[row] - o0;
          lsum += 0.5f * (s + res * res * e);
          d[0] = -res * e * inv_b;
          d[1] = in ? 0.5f * (1.0f - res * res * e) * inv_b : 0.0f;
        } else {
          const float Y = y[row], B1 = st_scale * st[row] + 1.0f;
          const float lam = B1 * __expf(fminf(o0, 30.0f));
          const float q = log1pf(Y) - log1pf(lam);
          lsum += (lam - Y * __logf(lam)) / B1 + 0.5f * (s + q * q * e);
          d[0] = o0 < 30.0f ? (lam - Y) / B1 * inv_b : 0.0f;
          d[1] = in ? 0.5f * (1.0f - q * q * e) * inv_b : 0.0f;
        }
      }
      put8(S.O, gt, 0, kOutP, d);
#pragma unroll
      for (int o = 0; o < 8; ++o) S.OT[core_idx(o, gt, 128)] = __float2bfloat16(d[o]);
      d[0] = d[1] = 0.0f;
      put8(S.O, gt, 8, kOutP, d);
#pragma unroll
      for (int o = 8; o < kOutP; ++o) S.OT[core_idx(o, gt, 128)] = __float2bfloat16(0.0f);
    }
    // ---- layer 4: dZ3 = (dout W4) gelu'(Z3), dW4 = dout^T H3 (transposed)
    stage_ht(S.T0, zb, valid);
    ready();
    if (tid == 0) {
      gemm_tile(dc, S.O, S.W4T, kOutP, kH, false);
      mma_commit(&S.mbar);
    }
    wait();
    upstream(zb, valid, gp);
    put_rows(S.T1, gp);
    ready();
    if (tid == 0) {
      gemm_tile(ac, S.T0, S.OT, 128, kOutP, false);  // Z3's columns are free now
      gemm_tile(dc, S.T1, S.W3T, kH, kH, false);
      mma_commit(&S.mbar);
    }
    wait();
    if (g == 0) {
      uint32_t r[16];
      TL_TMEM_LD_X16(ac + lanes, r);
      tmem_wait_ld();
      for (int o = 0; o < 2; ++o) part_put(P + kOffW4 + o * kH + gt, __uint_as_float(r[o]), first);
      if (tid < 2) {
        float a = 0.0f;
        for (int k = 0; k < 128; ++k) a += __bfloat162float(S.OT[core_idx(tid, k, 128)]);
        part_put(P + kOffB4 + tid, a, first);
      }
    }
    // ---- layers 3 and 2: dW = G^T H of the layer below, then the next G
#pragma unroll 1
    for (int l = 1; l >= 0; --l) {
      load_z(l, zb);
      stage_gt(S.T0, gp);
      stage_ht(S.T1, zb, valid);
      ready();
      if (tid == 0) {
        gemm_tile(ac, S.T0, S.T1, 128, kH, false);
        mma_commit(&S.mbar);
      }
      upstream(zb, valid, gp);  // dc: (G W) of this layer, computed with the last wait
      bias_grad(S.T0, P + (l == 1 ? kOffB3 : kOffB2));
      wait();
      write_w(P + (l == 1 ? kOffW3 : kOffW2), kH);
      if (l == 1) {
        put_rows(S.T1, gp);
        ready();
        if (tid == 0) {
          gemm_tile(dc, S.T1, S.W2T, kH, kH, false);
          mma_commit(&S.mbar);
        }
        wait();
      }
    }
    // ---- layer 1: dW1 = G1^T X
    __syncthreads();  // the bias gradient has read T0
    stage_gt(S.T0, gp);
    {
      float v[8];
      features8(x, row, valid, S.w.norm, 8 * g, v);
#pragma unroll
      for (int j = 0; j < 8; ++j) S.T1[core_idx(8 * g + j, gt, 128)] = __float2bfloat16(v[j]);
    }
    ready();
    if (tid == 0) {
      gemm_tile(ac, S.T0, S.T1, 128, kInP, false);
      mma_commit(&S.mbar);
    }
    bias_grad(S.T0, P + kOffB1);
    wait();
    write_w(P + kOffW1, kIn);
    tc_fence_before();
    __syncthreads();  // tiles and accumulators are free for the next tile
    tc_fence_after();
    first = false;
  }
  if (g == 0) {
    for (int off = 16; off; off >>= 1) lsum += __shfl_xor_sync(0xffffffffu, lsum, off);
    if ((tid & 31) == 0) S.loss[warp] = lsum;
  }
  if (!ok) set_error(err);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (tid == 0) part_loss[blockIdx.x] = (S.loss[0] + S.loss[1]) + (S.loss[2] + S.loss[3]);
  if (warp == 0) tmem_dealloc(tm, 512);
}

// grad[p] = sum over the blocks b (in order) of part[b * kParams + p]: every
// block writes every parameter's entry of its slice; and the loss likewise
__global__ void __launch_bounds__(256) k_mlp_wsum(const float *__restrict__ part,
                                                  const float *__restrict__ part_loss, int blocks,
                                                  float *grad, float *loss) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p == 0) {
    float a = 0.0f;
    for (int b = 0; b < blocks; ++b) a += part_loss[b];
    *loss = a;
  }
  if (p >= kParams) return;
  float acc = 0.0f;
#pragma unroll 8
  for (int b = 0; b < blocks; ++b) acc += part[(size_t)b * kParams + p];
  grad[p] = acc;
}

// ---------------------------------------------------------------- optimiser

// AdamW on the flat FP32 parameters (bias-corrected moments, decoupled decay
// on weights only).
__global__ void k_adamw(float *prm, const float *grad, float *m, float *v, int n, float lr,
                        float b1, float b2, float eps, float wd, float c1, float c2) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= n) return;
  const float g = grad[t];
  const float mt = b1 * m[t] + (1.0f - b1) * g;
  const float vt = b2 * v[t] + (1.0f - b2) * g * g;
  m[t] = mt;
  v[t] = vt;
  const bool is_bias = (t >= kOffB1 && t < kOffW2) || (t >= kOffB2 && t < kOffW3) ||
                       (t >= kOffB3 && t < kOffW4) || t >= kOffB4;
  float p = prm[t];
  if (!is_bias) p -= lr * wd * p;
  p -= lr * (mt / c1) / (sqrtf(vt / c2) + eps);
  prm[t] = p;
}

// ---------------------------------------------------------------- host side

static_assert(offsetof(FwdSmem, A) % 128 == 0 && offsetof(GradSmem, W2T) % 128 == 0 &&
                  offsetof(GradSmem, T0) % 128 == 0 && offsetof(GradSmem, OT) % 128 == 0 &&
                  offsetof(FwdSmem, mbar) % 8 == 0 && offsetof(GradSmem, mbar) % 8 == 0,
              "operand tiles are aligned");
constexpr size_t kFwdSmem = sizeof(FwdSmem) + 1024, kGradSmem = sizeof(GradSmem) + 1024;
static_assert(kFwdSmem <= 232448 && kGradSmem <= 232448, "227 KB of shared memory per block");

cudaError_t mlp_prepare() {
  cudaError_t e = cudaFuncSetAttribute(k_mlp_forward, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)kFwdSmem);
  if (e) return e;
  return cudaFuncSetAttribute(k_mlp_grad, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              (int)kGradSmem);
}

static int grad_blocks(int64_t M, int sms) {
  const int64_t tiles = (M + 127) / 128;
  return (int)(tiles < sms ? tiles : sms);
}

size_t mlp_grad_floats(int64_t M, int sms) {
  return (size_t)grad_blocks(M, sms) * (kParams + 1);
}

cudaError_t mlp_forward(const float *prm, const float *norm, const float *x, int64_t M, float *out,
                        int sms, int *err, long long spin, cudaStream_t s) {
  if (M <= 0) return cudaSuccess;
  k_mlp_forward<<<grad_blocks(M, sms), kThreads, kFwdSmem, s>>>(prm, norm, x, M, out, err, spin);
  return cudaGetLastError();
}

// loss and gradient of the mean loss over M rows; part: mlp_grad_floats(M, sms) floats
cudaError_t mlp_grad(const float *prm, const float *norm, const float *x, const float *y, int64_t M,
                     int sms, float *part, float *grad, float *loss, int *err, long long spin,
                     cudaStream_t s, int kind, const float *st, float st_scale) {
  const int g = grad_blocks(M, sms);
  float *part_loss = part + (size_t)g * kParams;
  k_mlp_grad<<<g, kThreads, kGradSmem, s>>>(prm, norm, x, y, M, part, part_loss, 1.0f / (float)M,
                                            err, spin, kind, st, st_scale);
  cudaError_t e = cudaGetLastError();
  if (e) return e;
  k_mlp_wsum<<<(kParams + 255) / 256, 256, 0, s>>>(part, part_loss, g, grad, loss);
  return cudaGetLastError();
}

cudaError_t mlp_adamw(float *prm, const float *grad, float *m, float *v, float lr, float wd,
                      int step, cudaStream_t s) {
  const float b1 = 0.9f, b2 = 0.999f;
  const float c1 = 1.0f - powf(b1, (float)step), c2 = 1.0f - powf(b2, (float)step);
  k_adamw<<<(kParams + 255) / 256, 256, 0, s>>>(prm, grad, m, v, kParams, lr, b1, b2, 1e-8f, wd,
                                                 c1, c2);
  return cudaGetLastError();
}

}  // namespace tl

// ---------------------------------------------------------------- C ABI

namespace {

std::mutex g_mu;

// Error words of the calls in flight: pinned host memory that a kernel writes only when
// a wait ran out, so that a call neither allocates, clears nor copies one.  One page,
// made on the first call; a call that finds no word free gets one of its own.
constexpr int kErrWords = 64;
int *g_err = nullptr;
unsigned long long g_err_used = 0;

int *err_take(int *slot) {
  std::lock_guard<std::mutex> lk(g_mu);
  *slot = -1;
  if (!g_err && cudaHostAlloc((void **)&g_err, sizeof(int) * kErrWords,
                              cudaHostAllocPortable | cudaHostAllocMapped) != cudaSuccess)
    g_err = nullptr;
  if (g_err)
    for (int q = 0; q < kErrWords; ++q)
      if (!(g_err_used >> q & 1ull)) {
        g_err_used |= 1ull << q;
        *slot = q;
        g_err[q] = 0;
        return g_err + q;
      }
  int *p = nullptr;
  if (cudaHostAlloc((void **)&p, sizeof(int), cudaHostAllocPortable | cudaHostAllocMapped) !=
      cudaSuccess)
    return nullptr;
  *p = 0;
  return p;
}

void err_give(int *p, int slot) {
  if (slot < 0) {
    cudaFreeHost(p);
    return;
  }
  std::lock_guard<std::mutex> lk(g_mu);
  g_err_used &= ~(1ull << slot);
}

// Per device, once: kernel attributes, the SM count, and a memory pool that keeps up to
// 64 MB of freed workspace (two calls' worth of the largest) instead of giving every
// call's back to the system.  Allocation and release are ordered on the call's stream.
struct Dev {
  bool ready = false;
  int sms = 0;
  cudaMemPool_t pool = nullptr;
};
Dev g_dev[64];

cudaError_t device(Dev *out) {
  int id = 0;
  cudaError_t e = cudaGetDevice(&id);
  if (e) return e;
  if (id < 0 || id >= 64) return cudaErrorInvalidDevice;
  std::lock_guard<std::mutex> lk(g_mu);
  Dev &d = g_dev[id];
  if (!d.ready) {
    if ((e = tl::mlp_prepare())) return e;
    if ((e = cudaDeviceGetAttribute(&d.sms, cudaDevAttrMultiProcessorCount, id))) return e;
    if (!d.pool) {
      cudaMemPoolProps pr;
      memset(&pr, 0, sizeof(pr));
      pr.allocType = cudaMemAllocationTypePinned;
      pr.location.type = cudaMemLocationTypeDevice;
      pr.location.id = id;
      if ((e = cudaMemPoolCreate(&d.pool, &pr))) return e;
      unsigned long long keep = 64ull << 20;
      if ((e = cudaMemPoolSetAttribute(d.pool, cudaMemPoolAttrReleaseThreshold, &keep))) return e;
    }
    d.ready = true;
  }
  *out = d;
  return cudaSuccess;
}

}  // namespace

extern "C" int trilens_mlp_forward(const float *params, const float *norm, const float *x,
                                   int64_t m, float *out, trilens_stream_t stream) {
  if (!params || !norm || m < 0 || (m > 0 && (!x || !out))) return TRILENS_ERR_INVALID;
  cudaStream_t s = (cudaStream_t)stream;
  Dev d;
  if (device(&d)) return TRILENS_ERR_CUDA;
  int slot;
  int *err = err_take(&slot);
  if (!err) return TRILENS_ERR_CUDA;
  int rc = TRILENS_OK;
  if (tl::mlp_forward(params, norm, x, m, out, d.sms, err, 1ll << 24, s) ||
      cudaStreamSynchronize(s))
    rc = TRILENS_ERR_CUDA;
  else if (*(volatile int *)err)
    rc = TRILENS_ERR_TIMEOUT;
  err_give(err, slot);
  return rc;
}

extern "C" int trilens_mlp_grad(const float *params, const float *norm, const float *x,
                                const float *y, const float *st, float st_scale, int32_t loss_kind,
                                int64_t m, float *grad, float *loss, trilens_stream_t stream) {
  if (!params || !norm || !grad || !loss || m < 1 || !x || !y) return TRILENS_ERR_INVALID;
  if (loss_kind != 0 && (loss_kind != 1 || !st)) return TRILENS_ERR_INVALID;
  cudaStream_t s = (cudaStream_t)stream;
  Dev d;
  if (device(&d)) return TRILENS_ERR_CUDA;
  int slot;
  int *err = err_take(&slot);
  if (!err) return TRILENS_ERR_CUDA;
  float *part = nullptr;
  int rc = TRILENS_OK;
  if (cudaMallocFromPoolAsync((void **)&part, sizeof(float) * tl::mlp_grad_floats(m, d.sms), d.pool,
                              s) != cudaSuccess) {
    rc = TRILENS_ERR_CUDA;
  } else {
    if (tl::mlp_grad(params, norm, x, y, m, d.sms, part, grad, loss, err, 1ll << 24, s, loss_kind,
                     st, st_scale))
      rc = TRILENS_ERR_CUDA;
    cudaFreeAsync(part, s);
    if (cudaStreamSynchronize(s)) rc = TRILENS_ERR_CUDA;
    else if (rc == TRILENS_OK && *(volatile int *)err) rc = TRILENS_ERR_TIMEOUT;
  }
  err_give(err, slot);
  return rc;
}
