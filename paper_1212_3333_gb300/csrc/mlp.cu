// MLP kernels of the learned segment proposal: packing, tensor-core inference, training
// (loss + gradient) and Adam.  Declarations and contracts: include/amr.h.
#include <cstring>

#include "ctx.h"
#include "mlp.cuh"

static_assert(amr::kPackBytes == AMR_MLP_PACKED_BYTES, "packed MLP image size");
static_assert(amr::kMlpParams == AMR_MLP_PARAMS, "MLP parameter count");
static_assert(amr::kMlpIn == AMR_MLP_FEATURES, "MLP feature count");

namespace amr {
namespace {

__device__ __forceinline__ float bf16r(float x) { return __bfloat162float(__float2bfloat16_rn(x)); }

// FP32 master parameters -> inference image (BF16 weights, padded rows, FP32 biases)
__global__ void pack_kernel(const float* __restrict__ p, unsigned char* __restrict__ out) {
  const int tid = blockIdx.x * blockDim.x + threadIdx.x;
  __nv_bfloat16* w1 = reinterpret_cast<__nv_bfloat16*>(out + kPackW1);
  __nv_bfloat16* w2 = reinterpret_cast<__nv_bfloat16*>(out + kPackW2);
  __nv_bfloat16* w3 = reinterpret_cast<__nv_bfloat16*>(out + kPackW3);
  __nv_bfloat16* w4 = reinterpret_cast<__nv_bfloat16*>(out + kPackW4);
  float* b = reinterpret_cast<float*>(out + kPackB);
  if (tid < kMlpH * kStride1) {
    const int o = tid / kStride1, i = tid % kStride1;
    w1[tid] = __float2bfloat16_rn(i < kMlpIn ? p[kOffW1 + o * kMlpIn + i] : 0.0f);
  }
  if (tid < kMlpH * kStrideH) {
    const int o = tid / kStrideH, i = tid % kStrideH;
    w2[tid] = __float2bfloat16_rn(i < kMlpH ? p[kOffW2 + o * kMlpH + i] : 0.0f);
    w3[tid] = __float2bfloat16_rn(i < kMlpH ? p[kOffW3 + o * kMlpH + i] : 0.0f);
  }
  if (tid < 8 * kStrideH) {
    const int o = tid / kStrideH, i = tid % kStrideH;
    w4[tid] = __float2bfloat16_rn(o == 0 && i < kMlpH ? p[kOffW4 + i] : 0.0f);
  }
  if (tid < 3 * kMlpH + 4) {
    float v = 0.0f;
    if (tid < kMlpH) v = p[kOffB1 + tid];
    else if (tid < 2 * kMlpH) v = p[kOffB2 + tid - kMlpH];
    else if (tid < 3 * kMlpH) v = p[kOffB3 + tid - 2 * kMlpH];
    else if (tid == 3 * kMlpH) v = p[kOffB4];
    b[tid] = v;
  }
}

// Inference on n rows of 12 features through the same warp routine the march uses.
__global__ void __launch_bounds__(128) forward_kernel(const unsigned char* __restrict__ packed,
                                                      const float* __restrict__ x, int64_t n,
                                                      float* __restrict__ y) {
  extern __shared__ __align__(16) unsigned char sm[];
  unsigned char* wsm = sm;
  for (int k = threadIdx.x; k < kPackBytes / 16; k += blockDim.x)
    reinterpret_cast<uint4*>(wsm)[k] = reinterpret_cast<const uint4*>(packed)[k];
  __syncthreads();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  __nv_bfloat16* xs = reinterpret_cast<__nv_bfloat16*>(sm + kPackBytes) + warp * 32 * kStride1;
  float* ys = reinterpret_cast<float*>(sm + kPackBytes + 4 * 32 * kStride1 * 2) + warp * 32;
  const int64_t tiles = (n + 31) / 32;
  for (int64_t tile = (int64_t)blockIdx.x * 4 + warp; tile < tiles; tile += (int64_t)gridDim.x * 4) {
    const int64_t r = tile * 32 + lane;
#pragma unroll
    for (int k = 0; k < kMlpInPad; ++k)
      xs[lane * kStride1 + k] = __float2bfloat16_rn(r < n && k < kMlpIn ? x[r * kMlpIn + k] : 0.0f);
    __syncwarp();
    const float v = mlp_forward_warp(wsm, xs, ys, lane);
    if (r < n) y[r] = v;
    __syncwarp();
  }
}

// Loss and gradient on the tensor cores (mma.sync.m16n8k16, BF16 x BF16 -> FP32), tiles of 128
// rows, 16 rows per warp.  The forward rounds weights and activations to BF16 exactly as
// inference does.  Every product of the backward has one operand that is a BF16 value already
// (a weight, an activation, a feature); the other, a delta in FP32, enters as the sum of three
// BF16 values (8 + 8 + 8 bits of its 24), so products are those of FP32.  The tensor cores
// round their FP32 sums toward zero, which adds up along a chain of them, so every 16 products
// (all three parts) start from zero and are added to the running sum by an FP32 addition:
// error of the gradient against 64 bits, median of 12 seeds, FP32 chains of one thread per row /
// this: batch 300 1.1e-7 / 5.7e-8, 4999 5.8e-7 / 8.0e-8, 16384 4.0e-7 / 1.4e-7, 131072 7.4e-7 / 1.4e-7
// (chained products, two seeds at 16384: 7.0e-7 / 1.2e-6).  A step (gradient, reduction, Adam) of 16384
// rows takes 33 us against 131 for one thread per row on the CUDA cores, of 131072 rows 99
// against 783 us; at 16384 rows and below its latencies bound it (one tile per block).
// Activations and deltas of the tile lie in shared memory for the weight gradients, whose
// 64 x 64 outputs the eight warps share (16 x 32 each, the tile's 128 rows in order); column
// kMlpH of the activations (kMlpIn of the features) holds ones, whose gradient is the bias's.
constexpr int kGradRows = 128;
constexpr int kGradThreads = 256;
struct GradShared {
  __nv_bfloat16 act[3][kGradRows][kStrideH];     // A1..A3; column kMlpH: 1, then 0
  __nv_bfloat16 delta[2][3][kGradRows][kStrideH];  // two layers' deltas in three parts
  __nv_bfloat16 x[kGradRows][kStride1];          // features; column kMlpIn: 1, then 0
  __nv_bfloat16 w1[kMlpH][kStride1];
  __nv_bfloat16 w[2][kMlpH][kStrideH];           // W2, W3
  __nv_bfloat16 d4[3][kGradRows];                // output deltas in three parts
  float b[3][kMlpH], w4[kMlpH], b4;
  float loss[kGradThreads / 32];
};

__device__ __forceinline__ void ldmatrix4_trans(uint32_t (&r)[4], const __nv_bfloat16* p) {
  const uint32_t a = (uint32_t)__cvta_generic_to_shared(p);
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];\n"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(a) : "memory");
}
__device__ __forceinline__ void ldmatrix2_trans(uint32_t (&r)[2], const __nv_bfloat16* p) {
  const uint32_t a = (uint32_t)__cvta_generic_to_shared(p);
  asm volatile("ldmatrix.sync.aligned.m8n8.x2.trans.shared.b16 {%0,%1}, [%2];\n"
               : "=r"(r[0]), "=r"(r[1])
               : "r"(a) : "memory");
}

// (x0, x1) as three BF16 pairs whose sums are x0 and x1 to 24 bits.
__device__ __forceinline__ void split3(float x0, float x1, uint32_t (&p)[3]) {
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const __nv_bfloat162 h = __floats2bfloat162_rn(x0, x1);
    p[k] = *reinterpret_cast<const uint32_t*>(&h);
    const float2 f = __bfloat1622float2(h);
    x0 -= f.x;
    x1 -= f.y;
  }
}

// d += A B over 16 products, from zero.
template <int P>
__device__ __forceinline__ void mma_add(float (&d)[4], const uint32_t (*a)[4], int stride,
                                        uint32_t b0, uint32_t b1) {
  float c[4] = {0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll
  for (int k = P - 1; k >= 0; --k) mma_bf16(c, a[k * stride], b0, b1);
#pragma unroll
  for (int q = 0; q < 4; ++q) d[q] += c[q];
}

// acc += A W^T (forward): the warp's 16 rows, KS k-steps, weights [out][in] of row stride S.
template <int KS, int S>
__device__ __forceinline__ void grad_forward(const uint32_t (&a)[KS][4], const __nv_bfloat16 (*w)[S],
                                             const float* bias, int lane, float (&acc)[8][4]) {
  const int g = lane >> 2, t = lane & 3;
#pragma unroll
  for (int n = 0; n < 8; ++n) {
    acc[n][0] = acc[n][2] = bias[8 * n + 2 * t];
    acc[n][1] = acc[n][3] = bias[8 * n + 2 * t + 1];
    const uint32_t* row = reinterpret_cast<const uint32_t*>(w[8 * n + g]);
#pragma unroll
    for (int s = 0; s < KS; ++s)
      mma_add<1>(acc[n], &a[s], 0, row[8 * s + t], row[8 * s + 4 + t]);
  }
}

// ReLU and rounding of the accumulators: the next layer's A fragments, and the rows in
// shared memory.
__device__ __forceinline__ void grad_store_act(const float (&acc)[8][4], uint32_t (&a)[4][4],
                                               __nv_bfloat16 (*act)[kStrideH], int row, int t) {
#pragma unroll
  for (int s = 0; s < 4; ++s)
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int n = 2 * s + h;
      a[s][2 * h] = relu_bf16x2(acc[n][0], acc[n][1]);
      a[s][2 * h + 1] = relu_bf16x2(acc[n][2], acc[n][3]);
      *reinterpret_cast<uint32_t*>(&act[row][8 * n + 2 * t]) = a[s][2 * h];
      *reinterpret_cast<uint32_t*>(&act[row + 8][8 * n + 2 * t]) = a[s][2 * h + 1];
    }
}

// Deltas (the accumulators' layout) where the activation is positive, in three parts: A
// fragments p[part][k-step], and the rows in shared memory.
__device__ __forceinline__ void grad_store_delta(const float (&d)[8][4], uint32_t (&p)[3][4][4],
                                                 __nv_bfloat16 (*delta)[kGradRows][kStrideH],
                                                 int row, int t) {
#pragma unroll
  for (int n = 0; n < 8; ++n) {
    const int s = n >> 1, h = n & 1;
    uint32_t lo[3], hi[3];
    split3(d[n][0], d[n][1], lo);
    split3(d[n][2], d[n][3], hi);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      p[k][s][2 * h] = lo[k];
      p[k][s][2 * h + 1] = hi[k];
      *reinterpret_cast<uint32_t*>(&delta[k][row][8 * n + 2 * t]) = lo[k];
      *reinterpret_cast<uint32_t*>(&delta[k][row + 8][8 * n + 2 * t]) = hi[k];
    }
  }
}

// Deltas of the layer below: d = (p W) where its activations (A fragments a) are positive.
__device__ __forceinline__ void grad_backward(const uint32_t (&p)[3][4][4],
                                              const __nv_bfloat16 (*w)[kStrideH],
                                              const uint32_t (&a)[4][4], int lane,
                                              float (&d)[8][4]) {
#pragma unroll
  for (int n = 0; n < 8; ++n)
#pragma unroll
    for (int c = 0; c < 4; ++c) d[n][c] = 0.0f;
#pragma unroll
  for (int s = 0; s < 4; ++s)
#pragma unroll
    for (int n = 0; n < 8; n += 2) {
      uint32_t b[4];  // (k, n), (k + 8, n), (k, n + 8), (k + 8, n + 8)
      ldmatrix4_trans(b, &w[16 * s + (lane & 15)][8 * n + 8 * (lane >> 4)]);
      mma_add<3>(d[n], &p[0][s], 4, b[0], b[1]);
      mma_add<3>(d[n + 1], &p[0][s], 4, b[2], b[3]);
    }
#pragma unroll
  for (int n = 0; n < 8; ++n) {
    const float2 lo = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&a[n >> 1][2 * (n & 1)]));
    const float2 hi = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&a[n >> 1][2 * (n & 1) + 1]));
    d[n][0] = lo.x > 0.0f ? d[n][0] : 0.0f;
    d[n][1] = lo.y > 0.0f ? d[n][1] : 0.0f;
    d[n][2] = hi.x > 0.0f ? d[n][2] : 0.0f;
    d[n][3] = hi.y > 0.0f ? d[n][3] : 0.0f;
  }
}

// g += delta^T act over the tile's rows: outputs 16 m .. 16 m + 15, NT column tiles from n0.
template <int NT, int S>
__device__ __forceinline__ void grad_weights(const __nv_bfloat16 (*delta)[kGradRows][kStrideH],
                                             const __nv_bfloat16 (*act)[S], int m, int n0, int lane,
                                             float (&g)[NT][4]) {
  float acc[NT][4] = {};
#pragma unroll 2
  for (int r = 0; r < kGradRows; r += 16) {
    uint32_t a[3][4];  // (o, r), (o + 8, r), (o, r + 8), (o + 8, r + 8)
#pragma unroll
    for (int k = 0; k < 3; ++k)
      ldmatrix4_trans(a[k], &delta[k][r + (lane & 7) + 8 * (lane >> 4)][16 * m + 8 * ((lane >> 3) & 1)]);
#pragma unroll
    for (int n = 0; n < NT; ++n) {
      uint32_t b[2];
      ldmatrix2_trans(b, &act[r + (lane & 15)][8 * (n0 + n)]);
      mma_add<3>(acc[n], a, 1, b[0], b[1]);
    }
  }
#pragma unroll
  for (int n = 0; n < NT; ++n)
#pragma unroll
    for (int c = 0; c < 4; ++c) g[n][c] += acc[n][c];
}

// One block's gradient entries of a weight matrix [64][ni] at offset w and its biases at b
// (the columns from ni on), from fragments of column tile n.
__device__ __forceinline__ void grad_write(float* part, const float (&c)[4], int w, int b, int ni,
                                           int m, int n, int lane) {
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int o = 16 * m + (lane >> 2) + 8 * (q >> 1), i = 8 * n + 2 * (lane & 3) + (q & 1);
    if (i < ni) part[w + o * ni + i] = c[q];
    else if (i == ni) part[b + o] = c[q];
  }
}

__global__ void __launch_bounds__(kGradThreads, 1)
    grad_kernel(const float* __restrict__ params, const float* __restrict__ x,
                const float* __restrict__ tgt, int64_t n_total, int64_t first, int64_t n,
                int64_t perm_a, int64_t perm_b, float* __restrict__ partial,
                float* __restrict__ loss_part) {
  extern __shared__ __align__(16) unsigned char raw[];
  GradShared& S = *reinterpret_cast<GradShared*>(raw);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int g = lane >> 2, t = lane & 3;
  // weights as BF16 (padding columns zero), biases FP32, the columns of ones
  for (int k = tid; k < kMlpH * kStride1; k += kGradThreads) {
    const int o = k / kStride1, i = k % kStride1;
    S.w1[o][i] = __float2bfloat16_rn(i < kMlpIn ? params[kOffW1 + o * kMlpIn + i] : 0.0f);
  }
  for (int k = tid; k < kMlpH * kMlpH; k += kGradThreads) {
    S.w[0][k / kMlpH][k % kMlpH] = __float2bfloat16_rn(params[kOffW2 + k]);
    S.w[1][k / kMlpH][k % kMlpH] = __float2bfloat16_rn(params[kOffW3 + k]);
  }
  if (tid < kMlpH) {
    S.b[0][tid] = params[kOffB1 + tid];
    S.b[1][tid] = params[kOffB2 + tid];
    S.b[2][tid] = params[kOffB3 + tid];
    S.w4[tid] = bf16r(params[kOffW4 + tid]);
  }
  if (tid == 0) S.b4 = params[kOffB4];
  for (int k = tid; k < 3 * kGradRows * 8; k += kGradThreads)
    S.act[k / (kGradRows * 8)][k / 8 % kGradRows][kMlpH + k % 8] =
        __float2bfloat16_rn(k % 8 == 0 ? 1.0f : 0.0f);
  for (int k = tid; k < kGradRows * (kStride1 - kMlpIn); k += kGradThreads) {
    const int i = k % (kStride1 - kMlpIn);
    S.x[k / (kStride1 - kMlpIn)][kMlpIn + i] = __float2bfloat16_rn(i == 0 ? 1.0f : 0.0f);
  }
  __syncthreads();

  // this warp's share of the weight gradients: outputs 16 m .., column tiles 4 h .. (and the
  // column of ones, tile 8, for h = 1)
  const int m = warp & 3, h = warp >> 2;
  float g3[4][4] = {}, g2[4][4] = {}, gb3[1][4] = {}, gb2[1][4] = {}, g1[1][4] = {};
  float g4[2][4] = {};  // of W4: column tile `warp`, and tile 8 (the bias) in warp 0
  float loss = 0.0f;
  const float inv_n = 1.0f / (float)n;
  const int64_t tiles = (n + kGradRows - 1) / kGradRows;
  for (int64_t tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
    {  // two threads per row: features as BF16
      const int r = tid >> 1, half = tid & 1;
      const int64_t rb = tile * kGradRows + r;
      float2 f[3] = {};
      if (rb < n) {
        const int64_t row = (int64_t)((uint64_t)(perm_a * (first + rb) + perm_b) % (uint64_t)n_total);
        const float* p = x + row * kMlpIn + 6 * half;
#pragma unroll
        for (int k = 0; k < 3; ++k) f[k] = make_float2(p[2 * k], p[2 * k + 1]);
      }
      uint32_t* d = reinterpret_cast<uint32_t*>(&S.x[r][6 * half]);
#pragma unroll
      for (int k = 0; k < 3; ++k) d[k] = pack_bf16(f[k].x, f[k].y);
    }
    __syncwarp();  // (a warp reads back its own 16 rows only)
    const int row = 16 * warp + g;
    // the targets of rows `row` and `row + 8`
    float tv[2];
    bool valid[2];
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const int64_t rb = tile * kGradRows + row + 8 * q;
      valid[q] = rb < n;
      tv[q] = valid[q] ? tgt[(uint64_t)(perm_a * (first + rb) + perm_b) % (uint64_t)n_total] : 0.0f;
    }
    // ---- forward
    uint32_t a1[4][4], a2[4][4], a3[4][4];
    float acc[8][4];
    {
      uint32_t ax[1][4];
      const uint32_t* r0 = reinterpret_cast<const uint32_t*>(S.x[row]);
      const uint32_t* r8 = reinterpret_cast<const uint32_t*>(S.x[row + 8]);
      ax[0][0] = r0[t];
      ax[0][1] = r8[t];
      ax[0][2] = r0[4 + t];
      ax[0][3] = r8[4 + t];
      grad_forward<1, kStride1>(ax, S.w1, S.b[0], lane, acc);
    }
    grad_store_act(acc, a1, S.act[0], row, t);
    grad_forward<4, kStrideH>(a1, S.w[0], S.b[1], lane, acc);
    grad_store_act(acc, a2, S.act[1], row, t);
    grad_forward<4, kStrideH>(a2, S.w[1], S.b[2], lane, acc);
    grad_store_act(acc, a3, S.act[2], row, t);
    // ---- output, loss and output delta of rows `row` and `row + 8` (each in four lanes)
    float z[2] = {0.0f, 0.0f}, dz[2];
#pragma unroll
    for (int c = 0; c < 8; ++c) {
      const float2 w4 = *reinterpret_cast<const float2*>(&S.w4[8 * c + 2 * t]);
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        const float2 v = __bfloat1622float2(
            *reinterpret_cast<const __nv_bfloat162*>(&a3[c >> 1][2 * (c & 1) + q]));
        z[q] = fmaf(v.x, w4.x, fmaf(v.y, w4.y, z[q]));
      }
    }
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      z[q] += __shfl_xor_sync(0xffffffffu, z[q], 1);
      z[q] += __shfl_xor_sync(0xffffffffu, z[q], 2);
      z[q] += S.b4;
      const float y = 1.0f / (1.0f + expf(-z[q]));
      if (valid[q] && t == 0) {
        const float sp = z[q] > 0.0f ? z[q] + log1pf(expf(-z[q])) : log1pf(expf(z[q]));
        loss += sp - tv[q] * z[q];
      }
      dz[q] = valid[q] ? (y - tv[q]) * inv_n : 0.0f;
    }
    if (t == 0) {
      uint32_t d[3];
      split3(dz[0], dz[1], d);
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        const __nv_bfloat162 v = *reinterpret_cast<const __nv_bfloat162*>(&d[k]);
        S.d4[k][row] = v.x;
        S.d4[k][row + 8] = v.y;
      }
    }
    // ---- delta of layer 3
#pragma unroll
    for (int c = 0; c < 8; ++c) {
      const float2 w4 = *reinterpret_cast<const float2*>(&S.w4[8 * c + 2 * t]);
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        const float2 v = __bfloat1622float2(
            *reinterpret_cast<const __nv_bfloat162*>(&a3[c >> 1][2 * (c & 1) + q]));
        acc[c][2 * q] = v.x > 0.0f ? dz[q] * w4.x : 0.0f;
        acc[c][2 * q + 1] = v.y > 0.0f ? dz[q] * w4.y : 0.0f;
      }
    }
    uint32_t p[3][4][4];
    grad_store_delta(acc, p, S.delta[0], row, t);
    __syncthreads();
    // ---- weight gradients of layers 4 and 3, delta of layer 2
    {
      float c4[2][4] = {};
#pragma unroll
      for (int r = 0; r < kGradRows; r += 16) {
        uint32_t b[2], b8[2] = {0, 0};
        ldmatrix2_trans(b, &S.act[2][r + (lane & 15)][8 * warp]);
        if (warp == 0) ldmatrix2_trans(b8, &S.act[2][r + (lane & 15)][kMlpH]);
        uint32_t a[3][4];  // row 0 of the A tile is the output delta
#pragma unroll
        for (int k = 0; k < 3; ++k) {
          const uint32_t* d = reinterpret_cast<const uint32_t*>(&S.d4[k][r]);
          a[k][0] = g == 0 ? d[t] : 0u;
          a[k][2] = g == 0 ? d[4 + t] : 0u;
          a[k][1] = a[k][3] = 0u;
        }
        mma_add<3>(c4[0], a, 1, b[0], b[1]);
        if (warp == 0) mma_add<3>(c4[1], a, 1, b8[0], b8[1]);
      }
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        g4[0][q] += c4[0][q];
        g4[1][q] += c4[1][q];
      }
    }
    grad_weights<4, kStrideH>(S.delta[0], S.act[1], m, 4 * h, lane, g3);
    if (h == 1) grad_weights<1, kStrideH>(S.delta[0], S.act[1], m, 8, lane, gb3);
    grad_backward(p, S.w[1], a2, lane, acc);
    grad_store_delta(acc, p, S.delta[1], row, t);
    __syncthreads();
    // ---- weight gradients of layer 2, delta of layer 1
    grad_weights<4, kStrideH>(S.delta[1], S.act[0], m, 4 * h, lane, g2);
    if (h == 1) grad_weights<1, kStrideH>(S.delta[1], S.act[0], m, 8, lane, gb2);
    grad_backward(p, S.w[0], a1, lane, acc);
    grad_store_delta(acc, p, S.delta[0], row, t);
    __syncthreads();
    // ---- weight gradients of layer 1
    grad_weights<1, kStride1>(S.delta[0], S.x, m, h, lane, g1);
    __syncthreads();  // the next tile overwrites the features and activations
  }
  // this block's partial sums, reduced over the blocks in a fixed order by reduce_kernel
  // (no atomics: the gradient is the same bit for bit on every call)
  float* part = partial + (size_t)blockIdx.x * kMlpParams;
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    grad_write(part, g3[c], kOffW3, kOffB3, kMlpH, m, 4 * h + c, lane);
    grad_write(part, g2[c], kOffW2, kOffB2, kMlpH, m, 4 * h + c, lane);
  }
  if (h == 1) {
    grad_write(part, gb3[0], kOffW3, kOffB3, kMlpH, m, 8, lane);
    grad_write(part, gb2[0], kOffW2, kOffB2, kMlpH, m, 8, lane);
  }
  grad_write(part, g1[0], kOffW1, kOffB1, kMlpIn, m, h, lane);
  if (g == 0) {
    part[kOffW4 + 8 * warp + 2 * t] = g4[0][0];
    part[kOffW4 + 8 * warp + 2 * t + 1] = g4[0][1];
    if (warp == 0 && t == 0) part[kOffB4] = g4[1][0];
  }
  for (int off = 16; off > 0; off >>= 1) loss += __shfl_down_sync(0xffffffffu, loss, off);
  if (lane == 0) S.loss[warp] = loss;
  __syncthreads();
  if (tid == 0) {
    float s = 0.0f;
    for (int w = 0; w < kGradThreads / 32; ++w) s += S.loss[w];
    loss_part[blockIdx.x] = s * inv_n;
  }
}

// grad[k] = sum of the blocks' partials in a fixed order: four runs of consecutive blocks,
// each by a thread of its own, then the runs in pairs; loss likewise (k = kMlpParams).
constexpr int kReduceCols = 64;
__global__ void __launch_bounds__(4 * kReduceCols)
    reduce_kernel(const float* __restrict__ partial, const float* __restrict__ loss_part,
                  int blocks, float* __restrict__ grad, float* __restrict__ loss) {
  __shared__ float run[4][kReduceCols];
  const int col = threadIdx.x % kReduceCols, q = threadIdx.x / kReduceCols;
  const int k = blockIdx.x * kReduceCols + col;
  const int lo = blocks * q / 4, hi = blocks * (q + 1) / 4;
  float s = 0.0f;
  if (k < kMlpParams) {
#pragma unroll 8
    for (int b = lo; b < hi; ++b) s += partial[(size_t)b * kMlpParams + k];
  } else if (k == kMlpParams) {
    for (int b = lo; b < hi; ++b) s += loss_part[b];
  }
  run[q][col] = s;
  __syncthreads();
  if (q == 0 && k <= kMlpParams) {
    s = (run[0][col] + run[1][col]) + (run[2][col] + run[3][col]);
    if (k < kMlpParams) grad[k] = s;
    else loss[0] = s;
  }
}

__global__ void adam_kernel(float* __restrict__ p, const float* __restrict__ g,
                            float* __restrict__ m, float* __restrict__ v, int n, float lr,
                            float b1, float b2, float eps, float c1, float c2) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= n) return;
  const float gk = g[k];
  const float mk = fmaf(b1, m[k], (1.0f - b1) * gk);
  const float vk = fmaf(b2, v[k], (1.0f - b2) * gk * gk);
  m[k] = mk;
  v[k] = vk;
  p[k] -= lr * (mk * c1) / (sqrtf(vk * c2) + eps);
}

thread_local std::string g_mlp_error;

amr_status mlp_fail(amr_status s, const std::string& m) {
  g_mlp_error = m;
  return s;
}

}  // namespace

const char* mlp_last_error() { return g_mlp_error.c_str(); }

}  // namespace amr

using namespace amr;

extern "C" {

amr_status amr_mlp_pack(const float* params_dev, void* packed_dev, void* stream) {
  if (!params_dev || !packed_dev || ((uintptr_t)packed_dev & 15))
    return mlp_fail(AMR_ERR_ARG, "params / packed buffer NULL or packed not 16-byte aligned");
  pack_kernel<<<(kMlpH * kStrideH + 255) / 256, 256, 0, (cudaStream_t)stream>>>(
      params_dev, (unsigned char*)packed_dev);
  cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? AMR_OK : mlp_fail(AMR_ERR_CUDA, cudaGetErrorString(e));
}

amr_status amr_mlp_forward(const void* packed_dev, const float* x_dev, int64_t n, float* y_dev,
                           void* stream) {
  if (!packed_dev || !x_dev || !y_dev || n < 0 || ((uintptr_t)packed_dev & 15))
    return mlp_fail(AMR_ERR_ARG, "bad MLP forward arguments");
  if (n == 0) return AMR_OK;
  const size_t smem = kPackBytes + 4 * 32 * kStride1 * 2 + 4 * 32 * 4;
  const int64_t tiles = (n + 31) / 32;
  const int blocks = (int)std::min<int64_t>((tiles + 3) / 4, 152 * 8);
  forward_kernel<<<blocks, 128, smem, (cudaStream_t)stream>>>((const unsigned char*)packed_dev,
                                                              x_dev, n, y_dev);
  cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? AMR_OK : mlp_fail(AMR_ERR_CUDA, cudaGetErrorString(e));
}

amr_status amr_mlp_loss_grad(const float* params_dev, const float* x_dev, const float* t_dev,
                             int64_t n_total, int64_t first, int64_t n, int64_t perm_a,
                             int64_t perm_b, float* grad_dev, float* loss_dev, float* scratch_dev,
                             void* stream) {
  if (!params_dev || !x_dev || !t_dev || !grad_dev || !loss_dev || !scratch_dev || n <= 0 ||
      n_total <= 0 ||
      first < 0 || perm_a <= 0 || perm_b < 0 || perm_a >= ((int64_t)1 << 31) ||
      n_total >= ((int64_t)1 << 31) || first + n >= ((int64_t)1 << 32))
    return mlp_fail(AMR_ERR_ARG, "bad MLP gradient arguments");
  cudaStream_t st = (cudaStream_t)stream;
  cudaError_t e = cudaFuncSetAttribute(grad_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)sizeof(GradShared));
  if (e != cudaSuccess) return mlp_fail(AMR_ERR_CUDA, cudaGetErrorString(e));
  const int64_t tiles = (n + kGradRows - 1) / kGradRows;
  const int blocks = (int)std::min<int64_t>(tiles, AMR_MLP_GRAD_BLOCKS);
  float* partial = scratch_dev;                                        // [blocks][params]
  float* loss_part = scratch_dev + (size_t)AMR_MLP_GRAD_BLOCKS * kMlpParams;  // [blocks]
  grad_kernel<<<blocks, kGradThreads, sizeof(GradShared), st>>>(params_dev, x_dev, t_dev, n_total, first,
                                                       n, perm_a, perm_b % n_total, partial,
                                                       loss_part);
  reduce_kernel<<<(kMlpParams + kReduceCols) / kReduceCols, 4 * kReduceCols, 0, st>>>(partial, loss_part, blocks, grad_dev,
                                                             loss_dev);
  e = cudaGetLastError();
  return e == cudaSuccess ? AMR_OK : mlp_fail(AMR_ERR_CUDA, cudaGetErrorString(e));
}

amr_status amr_mlp_adam(float* params_dev, const float* grad_dev, float* m_dev, float* v_dev,
                        float lr, float beta1, float beta2, float eps, int32_t step, void* stream) {
  if (!params_dev || !grad_dev || !m_dev || !v_dev || step < 1)
    return mlp_fail(AMR_ERR_ARG, "bad Adam arguments");
  const float c1 = 1.0f / (1.0f - powf(beta1, (float)step));
  const float c2 = 1.0f / (1.0f - powf(beta2, (float)step));
  adam_kernel<<<(kMlpParams + 255) / 256, 256, 0, (cudaStream_t)stream>>>(
      params_dev, grad_dev, m_dev, v_dev, kMlpParams, lr, beta1, beta2, eps, c1, c2);
  cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? AMR_OK : mlp_fail(AMR_ERR_CUDA, cudaGetErrorString(e));
}

}  // extern "C"
