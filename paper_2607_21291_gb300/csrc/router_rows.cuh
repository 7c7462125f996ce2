// Hidden units of the router (Sec. 3.4) on CUDA cores: u = W1 x for a tile of
// 16 rows and 64 hidden units, fp32 accumulation of exact products. Shared by
// the fp32 router scores and the router's gradient.
//
// The contraction is small (64 outputs a row), so what bounds it is how often
// operands are read from shared memory and how many threads share a row: the
// 8 warps of a block each take every eighth 64-byte piece of the feature axis
// (a row of 512 fp32 features is 4 pieces a warp), transpose their pieces of x
// and W1 into shared memory of their own (no block barrier in the loop, the
// next piece already in flight in registers), and hold 4 rows x 8 units per
// thread: three 16-byte shared loads feed 32 multiply-adds. The warps' partial
// tiles are then added in warp order (bit-reproducible).
#pragma once

#include "common.cuh"

namespace adadsf {

constexpr int kRrRows = 16;        // rows of a block
constexpr int kRrUnits = 64;       // hidden units of a tile
constexpr int kRrWarps = 8;
constexpr int kRrThreads = 32 * kRrWarps;

template <typename T>
struct RouterRows {
  static constexpr int KC = 64 / (int)sizeof(T);           // features of a piece (64 bytes of a row)
  static constexpr int WARP_FLOATS = KC * (kRrUnits + kRrRows);
  static constexpr int RED_FLOATS = kRrWarps * kRrRows * kRrUnits;
  static constexpr int SMEM_FLOATS = kRrWarps * WARP_FLOATS > RED_FLOATS ? kRrWarps * WARP_FLOATS : RED_FLOATS;
  static constexpr int SMEM_BYTES = SMEM_FLOATS * 4;
};

// u[row][unit] (no bias) of 4 consecutive units: thread t holds row t / 16 and
// units u0 + 4 (t % 16) ... + 3 (zero past h). xr: row (lane % 16) of the tile
// (any valid row for the ones past the end); w1 [h][d]; d a multiple of 64,
// rows 16-byte aligned. Block-wide: shared memory is reused, with barriers
// on both sides.
template <typename T>
__device__ __forceinline__ float4 router_rows_units(const T* xr, const T* w1, int u0, int h, int d, float* smem) {
  using R = RouterRows<T>;
  constexpr int V = Elem<T>::kVec, KC = R::KC;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  float* ws = smem + warp * R::WARP_FLOATS;   // [KC][64]
  float* xs = ws + KC * kRrUnits;             // [KC][16]
  const int rg = lane >> 3, ug = lane & 7;
  float acc[4][8];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 8; ++j) acc[i][j] = 0.f;
  const int n = d / KC;
  uint4 wv[8], xv[2];
  auto fetch = [&](int c) {
    const T* wp = w1 + (int64_t)c * KC;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int unit = u0 + lane + 32 * (i & 1);
      wv[i] = unit < h ? *reinterpret_cast<const uint4*>(wp + (int64_t)unit * d + (i >> 1) * V) : make_uint4(0, 0, 0, 0);
    }
#pragma unroll
    for (int i = 0; i < 2; ++i)
      xv[i] = *reinterpret_cast<const uint4*>(xr + (int64_t)c * KC + ((lane >> 4) + 2 * i) * V);
  };
  if (warp < n) fetch(warp);
  for (int c = warp; c < n; c += kRrWarps) {
    __syncwarp();
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      float f[V];
      unpack16(wv[i], f, T());
#pragma unroll
      for (int e = 0; e < V; ++e) ws[((i >> 1) * V + e) * kRrUnits + lane + 32 * (i & 1)] = f[e];
    }
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      float f[V];
      unpack16(xv[i], f, T());
#pragma unroll
      for (int e = 0; e < V; ++e) xs[(((lane >> 4) + 2 * i) * V + e) * kRrRows + (lane & 15)] = f[e];
    }
    if (c + kRrWarps < n) fetch(c + kRrWarps);
    __syncwarp();
#pragma unroll 8
    for (int k = 0; k < KC; ++k) {
      const float4 x4 = *reinterpret_cast<const float4*>(xs + k * kRrRows + rg * 4);
      const float4 wa = *reinterpret_cast<const float4*>(ws + k * kRrUnits + ug * 4);
      const float4 wb = *reinterpret_cast<const float4*>(ws + k * kRrUnits + 32 + ug * 4);
      const float xf[4] = {x4.x, x4.y, x4.z, x4.w};
      const float wf[8] = {wa.x, wa.y, wa.z, wa.w, wb.x, wb.y, wb.z, wb.w};
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 8; ++j) acc[i][j] = fmaf(xf[i], wf[j], acc[i][j]);
    }
  }
  __syncthreads();   // the partial tiles overlay the warps' operand areas
  float* red = smem + warp * kRrRows * kRrUnits;   // [warp][16][64]
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    float* p = red + (rg * 4 + i) * kRrUnits + ug * 4;
    *reinterpret_cast<float4*>(p) = make_float4(acc[i][0], acc[i][1], acc[i][2], acc[i][3]);
    *reinterpret_cast<float4*>(p + 32) = make_float4(acc[i][4], acc[i][5], acc[i][6], acc[i][7]);
  }
  __syncthreads();
  float4 u = make_float4(0.f, 0.f, 0.f, 0.f);
  const float* q = smem + (threadIdx.x >> 4) * kRrUnits + (threadIdx.x & 15) * 4;
#pragma unroll
  for (int w = 0; w < kRrWarps; ++w) {
    const float4 f = *reinterpret_cast<const float4*>(q + w * kRrRows * kRrUnits);
    u.x += f.x;
    u.y += f.y;
    u.z += f.z;
    u.w += f.w;
  }
  __syncthreads();
  return u;
}

// Sum over the 16 threads that share a row.
__device__ __forceinline__ float row16_sum(float v) {
#pragma unroll
  for (int o = 8; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

}  // namespace adadsf
