// The linear classifier in fp32 (class token -> logits of the ViT, pooled
// features -> logits of ResNet-50): logits[b, c] = y[b, :] . W[c, :] + bias[c],
// y a row of X, normalised first for the ViT (LayerNorm over the first d_true
// of d channels; the rest are zero padding).
//
// Two kernels, chosen by the batch (classifier_launch):
//  - tile: 32 images x 32 classes a CTA, the reduction split over its 8 warps
//    and summed in shared memory. A lane holds 8 images x 4 classes, so 12
//    float4 reads feed 64 packed multiply-adds, and three chunks of the rows
//    are in flight (read straight from the L2 the same tile takes 50 us: too
//    little in flight). 4 classes x 8 images a warp, each warp over the whole
//    reduction, read W 16 times and the images 32 times from the L2: 128
//    images x 1000 classes x 2048 34.8 -> 24.5 us, 256 x 1000 x 768 with the
//    LayerNorm 42.9 -> 34.6 (event pairs, ~5 us of it the events).
//  - small batches: a warp per class and a CTA per 8 classes, so that 1000
//    classes fill the chip, and the class's row of W in registers before the
//    wait for the kernel that writes X. One image x 1000 x 768 16.3 -> 10.1 us.
#pragma once
#include "common.h"
#include "ptx.cuh"

namespace elasto {

namespace classifier {

constexpr int TILE = 32;                      // images and classes of a CTA
constexpr int WARPS = 8;
constexpr int RED_LD = TILE + 1;              // padded row of the partial sums
constexpr int RED_FLOATS = WARPS * TILE * RED_LD;
constexpr int SMALL_IMGS = 8, SMALL_BATCH = 15;  // images a CTA of the small kernel; largest batch it runs

__device__ __forceinline__ float sum32(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// One warp, R rows at once: y = LayerNorm(x) * g + b over the first d_true of
// d <= 128 * NV channels (d % 4 == 0), zeros after them; LN = false copies the
// rows. Row r: x + r * xs -> y + r * ys; rows from `rows` on are not touched.
template <bool LN, int NV, int R>
__device__ __forceinline__ void prepare_rows(const float* __restrict__ x, size_t xs, float* __restrict__ y, size_t ys,
                                             int rows, int d, int d_true, const float* __restrict__ g,
                                             const float* __restrict__ b, int lane) {
  float4 v[R][NV];
#pragma unroll
  for (int r = 0; r < R; ++r)
#pragma unroll
    for (int i = 0; i < NV; ++i) {
      const int c = (i * 32 + lane) * 4;
      v[r][i] = r < rows && c < d ? *reinterpret_cast<const float4*>(x + r * xs + c) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
#pragma unroll
  for (int r = 0; r < R; ++r) {
    float mean = 0.0f, rstd = 1.0f;
    if constexpr (LN) {
      float s = 0.0f, ss = 0.0f;
#pragma unroll
      for (int i = 0; i < NV; ++i) {
        const float* e = &v[r][i].x;
#pragma unroll
        for (int k = 0; k < 4; ++k) s += (i * 32 + lane) * 4 + k < d_true ? e[k] : 0.0f;
      }
      mean = sum32(s) / d_true;
#pragma unroll
      for (int i = 0; i < NV; ++i) {
        const float* e = &v[r][i].x;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const float a = e[k] - mean;
          ss += (i * 32 + lane) * 4 + k < d_true ? a * a : 0.0f;
        }
      }
      rstd = rsqrtf(sum32(ss) / d_true + 1e-6f);
    }
#pragma unroll
    for (int i = 0; i < NV; ++i) {
      const int c = (i * 32 + lane) * 4;
      if (r >= rows || c >= d) continue;
      float4 o = v[r][i];
      if constexpr (LN) {
        float* e = &o.x;
#pragma unroll
        for (int k = 0; k < 4; ++k)
          e[k] = c + k < d_true ? (e[k] - mean) * rstd * __ldg(g + c + k) + __ldg(b + c + k) : 0.0f;
      }
      *reinterpret_cast<float4*>(y + r * ys + c) = o;
    }
  }
}

// grid (ceil(C / 8), ceil(B / 8)): classes along x, which alone reaches past
// 65535 blocks; 256 threads, 8 * d floats of shared memory.
template <bool LN, int NV>
__global__ void __launch_bounds__(256) small_kernel(const float* __restrict__ X, size_t row, int B, int d, int d_true,
                                                    const float* __restrict__ g, const float* __restrict__ bta,
                                                    const float* __restrict__ W, const float* __restrict__ bias, int C,
                                                    float* __restrict__ logits) {
  extern __shared__ float4 smem4[];
  float* sy = reinterpret_cast<float*>(smem4);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int b0 = blockIdx.y * SMALL_IMGS, nimg = min(SMALL_IMGS, B - b0);
  const int c = blockIdx.x * WARPS + warp;
  const float* wr = W + static_cast<size_t>(min(c, C - 1)) * d;
  float4 w[NV];
#pragma unroll
  for (int i = 0; i < NV; ++i) {
    const int k = (i * 32 + lane) * 4;
    w[i] = k < d ? __ldg(reinterpret_cast<const float4*>(wr + k)) : make_float4(0.f, 0.f, 0.f, 0.f);
  }
  const float bc = __ldg(bias + min(c, C - 1));
  pdl_wait();
  pdl_trigger();
  if (warp < nimg) prepare_rows<LN, NV, 1>(X + (b0 + warp) * row, 0, sy + warp * d, 0, 1, d, d_true, g, bta, lane);
  __syncthreads();
  if (c >= C) return;
  for (int i = 0; i < nimg; ++i) {
    float2 acc = make_float2(0.0f, 0.0f);
#pragma unroll
    for (int k = 0; k < NV; ++k) {
      const int e = (k * 32 + lane) * 4;
      if (e < d) {
        const float4 y = *reinterpret_cast<const float4*>(sy + i * d + e);
        acc = fma2(make_float2(w[k].x, w[k].y), make_float2(y.x, y.y), acc);
        acc = fma2(make_float2(w[k].z, w[k].w), make_float2(y.z, y.w), acc);
      }
    }
    const float v = sum32(acc.x + acc.y);
    if (lane == 0) logits[static_cast<size_t>(b0 + i) * C + c] = v + bc;
  }
}

constexpr int KC = 128;                       // reduction values of a staged chunk
constexpr int LDK = KC + 4;                   // padded staged row: neighbouring rows in other banks
constexpr int RING = 3;                       // chunks in flight

__device__ __forceinline__ void copy16(float* dst, const float* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_addr(dst)), "l"(src) : "memory");
}

// grid (ceil(B / 32), at most ceil(C / 32)), 256 threads: a CTA takes the class
// tiles blockIdx.y, blockIdx.y + gridDim.y, ... Chunks of KC values of a tile's
// 32 rows of W (and, without LN, of X) come through a ring of asynchronous
// copies; each warp reduces an eighth of every chunk for all 32 x 32 outputs.
// With LN the 32 normalised rows are in shared memory whole. d % 4 == 0.
template <bool LN>
__global__ void __launch_bounds__(256) tile_kernel(const float* __restrict__ X, size_t row, int B, int d, int d_true,
                                                   const float* __restrict__ g, const float* __restrict__ bta,
                                                   const float* __restrict__ W, const float* __restrict__ bias, int C,
                                                   float* __restrict__ logits) {
  constexpr int ROWS = LN ? TILE : 2 * TILE;  // staged rows: W, then X
  extern __shared__ float4 smem4[];
  float* ring = reinterpret_cast<float*>(smem4);
  float* sy = ring + RING * ROWS * LDK;
  float* red = ring;  // the partial sums, once the ring is done
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int b0 = blockIdx.x * TILE, nimg = min(TILE, B - b0);
  const int chunks = (d + KC - 1) / KC, ldy = d + 4;
  int c0 = blockIdx.y * TILE;
  auto fetch = [&](int q) {  // chunk q: 32 pieces of 16 bytes a row, a warp a row; zeros past d
    if (q < chunks) {
      float* dst = ring + q % RING * ROWS * LDK;
      const int k = q * KC + lane * 4;
#pragma unroll
      for (int i = 0; i < ROWS / WARPS; ++i) {
        const int r = i * WARPS + warp;
        const float* src = r < TILE ? W + static_cast<size_t>(min(c0 + r, C - 1)) * d
                                    : X + (b0 + min(r - TILE, nimg - 1)) * row;
        if (k < d)
          copy16(dst + r * LDK + lane * 4, src + k);
        else
          *reinterpret_cast<float4*>(dst + r * LDK + lane * 4) = make_float4(0.f, 0.f, 0.f, 0.f);
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  if constexpr (LN) {  // W does not depend on the kernel before
#pragma unroll
    for (int q = 0; q < RING - 1; ++q) fetch(q);
  }
  pdl_wait();
  pdl_trigger();
  if constexpr (LN) {
    for (int i = 2 * warp; i < nimg; i += 2 * WARPS)
      prepare_rows<true, 8, 2>(X + (b0 + i) * row, row, sy + i * ldy, ldy, nimg - i, d, d_true, g, bta, lane);
  } else {
#pragma unroll
    for (int q = 0; q < RING - 1; ++q) fetch(q);
  }
  const int li = lane >> 3, lj = lane & 7;  // images 4 i + li, classes 8 j + lj
  for (;;) {
    float2 acc[8][4];
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) acc[i][j] = make_float2(0.0f, 0.0f);
    for (int q = 0; q < chunks; ++q) {
      asm volatile("cp.async.wait_group %0;" ::"n"(RING - 2) : "memory");
      __syncthreads();  // chunk q (and at q = 0 the rows) landed; chunk q - 1 read by all
      fetch(q + RING - 1);
      const float* sw = ring + q % RING * ROWS * LDK;
#pragma unroll
      for (int h = 0; h < KC / WARPS; h += 4) {
        const int e = warp * (KC / WARPS) + h;
        if (LN && q * KC + e >= d) continue;  // (the rows are d long)
        float4 y[8], w[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) w[j] = *reinterpret_cast<const float4*>(sw + (8 * j + lj) * LDK + e);
#pragma unroll
        for (int i = 0; i < 8; ++i)
          y[i] = *reinterpret_cast<const float4*>(LN ? sy + min(4 * i + li, nimg - 1) * ldy + q * KC + e
                                                     : sw + (TILE + 4 * i + li) * LDK + e);
#pragma unroll
        for (int i = 0; i < 8; ++i)
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            acc[i][j] = fma2(make_float2(y[i].x, y[i].y), make_float2(w[j].x, w[j].y), acc[i][j]);
            acc[i][j] = fma2(make_float2(y[i].z, y[i].w), make_float2(w[j].z, w[j].w), acc[i][j]);
          }
      }
    }
    __syncthreads();  // the ring is read: it takes the partial sums
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j)
        red[(warp * TILE + 4 * i + li) * RED_LD + 8 * j + lj] = acc[i][j].x + acc[i][j].y;
    __syncthreads();
    const int c = c0 + lane;
    for (int i = warp; i < nimg; i += WARPS) {
      float v = 0.0f;
#pragma unroll
      for (int q = 0; q < WARPS; ++q) v += red[(q * TILE + i) * RED_LD + lane];
      if (c < C) logits[static_cast<size_t>(b0 + i) * C + c] = v + bias[c];
    }
    c0 += gridDim.y * TILE;
    if (c0 >= C) break;
    __syncthreads();  // the partial sums are read: the ring takes the next tile
#pragma unroll
    for (int q = 0; q < RING - 1; ++q) fetch(q);
  }
}
static_assert(RED_FLOATS <= RING * TILE * LDK, "the partial sums fit the ring");

inline size_t tile_smem(bool ln, int d) {
  return (RING * (ln ? 1 : 2) * TILE * LDK + (ln ? size_t(TILE) * (d + 4) : 0)) * sizeof(float);
}

// Shared-memory limits of the kernels for rows of up to d values.
template <bool LN, int NV>
cudaError_t init_attributes(int d) {
  cudaError_t e = cudaFuncSetAttribute(small_kernel<LN, NV>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       SMALL_IMGS * d * static_cast<int>(sizeof(float)));
  if (e != cudaSuccess) return e;
  return cudaFuncSetAttribute(tile_kernel<LN>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              static_cast<int>(tile_smem(LN, d)));
}

// X: the row of image b at X + b * row (row and d multiples of 4, 16-byte
// aligned); d <= 128 * NV.
template <bool LN, int NV>
cudaError_t launch(const float* X, size_t row, int B, int d, int d_true, const float* g, const float* b, const float* W,
                   const float* bias, int C, float* logits, cudaStream_t s) {
  if (B > SMALL_BATCH) {  // one wave: with LN every CTA normalises its 32 rows, so it keeps them for several class tiles
    const int gx = (B + TILE - 1) / TILE, gy = (C + TILE - 1) / TILE, most = num_sms() / gx;
    return launch_pdl(tile_kernel<LN>, dim3(gx, LN && most < gy ? (most > 1 ? most : 1) : gy), dim3(256),
                      tile_smem(LN, d), s, X, row, B, d, d_true, g, b, W, bias, C, logits);
  }
  return launch_pdl(small_kernel<LN, NV>, dim3((C + WARPS - 1) / WARPS, (B + SMALL_IMGS - 1) / SMALL_IMGS), dim3(256),
                    SMALL_IMGS * d * sizeof(float), s, X, row, B, d, d_true, g, b, W, bias, C, logits);
}

}  // namespace classifier

}  // namespace elasto
