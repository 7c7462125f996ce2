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
// thread: three 16-byte shared loads feed 32 multiply-adds. Four lanes load a
// row's piece (8 lines an instruction; a row per lane made 32 and kept the L1
// pipe at 80 %), and the columns of the transposed pieces are XOR-ed with 8
// times the loading lane's vector so that these stores spread over the banks.
// The warps' partial tiles are then added in warp order (bit-reproducible).
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
  static constexpr int MMA_BYTES = RED_FLOATS * 4;         // router_rows_partial
};

// u[row][unit] (no bias) of 4 consecutive units: thread t holds row t / 16 and
// units u0 + 4 (t % 16) ... + 3 (zero past h). xr0, xr1: rows lane / 4 and lane / 4
// + 8 of the tile (any valid row for the ones past the end); w1 [h][d]; d a
// multiple of 64, rows 16-byte aligned. Block-wide: shared memory is reused, with barriers
// on both sides.
template <typename T>
__device__ __forceinline__ float4 router_rows_units(const T* xr0, const T* xr1, const T* w1, int u0, int h, int d, float* smem) {
  using R = RouterRows<T>;
  constexpr int V = Elem<T>::kVec, KC = R::KC;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  float* ws = smem + warp * R::WARP_FLOATS;   // [KC][64]
  float* xs = ws + KC * kRrUnits;             // [KC][16]
  const int rg = lane >> 3, ug = lane & 7;
  float tot[4][8];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 8; ++j) tot[i][j] = 0.f;
  const int n = d / KC;
  uint4 wv[8], xv[2];
  const int lrow = lane >> 2, lvec = lane & 3;
  auto fetch = [&](int c) {
    const int64_t k = (int64_t)c * KC + lvec * V;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int unit = u0 + lrow + 8 * i;
      wv[i] = unit < h ? *reinterpret_cast<const uint4*>(w1 + (int64_t)unit * d + k) : make_uint4(0, 0, 0, 0);
    }
    xv[0] = *reinterpret_cast<const uint4*>(xr0 + k);
    xv[1] = *reinterpret_cast<const uint4*>(xr1 + k);
  };
  if (warp < n) fetch(warp);
  for (int c = warp; c < n; c += kRrWarps) {
    __syncwarp();
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      float f[V];
      unpack16(wv[i], f, T());
#pragma unroll
      for (int e = 0; e < V; ++e) ws[(lvec * V + e) * kRrUnits + ((lrow + 8 * i) ^ (8 * lvec))] = f[e];
    }
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      float f[V];
      unpack16(xv[i], f, T());
#pragma unroll
      for (int e = 0; e < V; ++e) xs[(lvec * V + e) * kRrRows + ((lrow + 8 * i) ^ (8 * (lvec & 1)))] = f[e];
    }
    if (c + kRrWarps < n) fetch(c + kRrWarps);
    __syncwarp();
    float acc[4][8];   // the piece's own sums (short chains of roundings), then added to the total
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 8; ++j) acc[i][j] = 0.f;
#pragma unroll 8
    for (int k = 0; k < KC; ++k) {
      const int sw = 8 * (k / V);   // this k's column swizzle
      const float4 x4 = *reinterpret_cast<const float4*>(xs + k * kRrRows + ((rg * 4) ^ (sw & 8)));
      const float4 wa = *reinterpret_cast<const float4*>(ws + k * kRrUnits + ((ug * 4) ^ sw));
      const float4 wb = *reinterpret_cast<const float4*>(ws + k * kRrUnits + ((32 + ug * 4) ^ sw));
      const float xf[4] = {x4.x, x4.y, x4.z, x4.w};
      const float wf[8] = {wa.x, wa.y, wa.z, wa.w, wb.x, wb.y, wb.z, wb.w};
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 8; ++j) acc[i][j] = fmaf(xf[i], wf[j], acc[i][j]);
    }
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 8; ++j) tot[i][j] += acc[i][j];
  }
  __syncthreads();   // the partial tiles overlay the warps' operand areas
  float* red = smem + warp * kRrRows * kRrUnits;   // [warp][16][64]
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    float* p = red + (rg * 4 + i) * kRrUnits + ug * 4;
    *reinterpret_cast<float4*>(p) = make_float4(tot[i][0], tot[i][1], tot[i][2], tot[i][3]);
    *reinterpret_cast<float4*>(p + 32) = make_float4(tot[i][4], tot[i][5], tot[i][6], tot[i][7]);
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

// The same contraction for bf16 operands on warp-level tensor products (m16n8k16):
// the 16 rows are the A operand and eight units a B operand, both loaded straight
// from memory (16 bytes a lane; the order of k inside a product is free as long as
// both operands agree). Products are exact; each 32 k are summed by the tensor core
// from zero and added to the total in fp32, so that its truncating accumulator
// never carries a long sum (the gradient's error against 64 bits is 1.4e-7 at 2048 rows
// of 2048 features, 7.9e-7 as serial fp32 sums).
//
// One piece of 32 features of the operands, in flight.
struct RouterPiece {
  uint4 w[8], xa, xb;
  __device__ __forceinline__ void load_w(const bf16* w1, int d, int c) {
    const int lane = threadIdx.x & 31;
    const int64_t k = (int64_t)c * 32 + (lane & 3) * 8;
#pragma unroll
    for (int i = 0; i < 8; ++i) w[i] = *reinterpret_cast<const uint4*>(w1 + (int64_t)(8 * i + (lane >> 2)) * d + k);
  }
  __device__ __forceinline__ void load_x(const bf16* xr0, const bf16* xr1, int c) {
    const int64_t k = (int64_t)c * 32 + (threadIdx.x & 3) * 8;
    xa = *reinterpret_cast<const uint4*>(xr0 + k);
    xb = *reinterpret_cast<const uint4*>(xr1 + k);
  }
};
// The sums over pieces [c_lo, c_hi), which the warps take in turn; `next` holds the
// weights of the warp's first piece (c_lo + warp) if there is one. Returns what
// router_rows_units returns; smem: RED_FLOATS floats.
__device__ __forceinline__ float4 router_rows_partial(const bf16* xr0, const bf16* xr1, const bf16* w1, int d, int c_lo,
                                                      int c_hi, RouterPiece& next, float* smem) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int gid = lane >> 2, tig = lane & 3;
  float tot[8][4];
#pragma unroll
  for (int i = 0; i < 8; ++i) tot[i][0] = tot[i][1] = tot[i][2] = tot[i][3] = 0.f;
  if (c_lo + warp < c_hi) next.load_x(xr0, xr1, c_lo + warp);
  for (int c = c_lo + warp; c < c_hi; c += kRrWarps) {
    const RouterPiece cur = next;
    if (c + kRrWarps < c_hi) {
      next.load_w(w1, d, c + kRrWarps);
      next.load_x(xr0, xr1, c + kRrWarps);
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      float p[4] = {0.f, 0.f, 0.f, 0.f};
      mma_16816(p, cur.xa.x, cur.xb.x, cur.xa.y, cur.xb.y, cur.w[i].x, cur.w[i].y);
      mma_16816(p, cur.xa.z, cur.xb.z, cur.xa.w, cur.xb.w, cur.w[i].z, cur.w[i].w);
#pragma unroll
      for (int e = 0; e < 4; ++e) tot[i][e] += p[e];
    }
  }
  float* red = smem + warp * kRrRows * kRrUnits;   // [warp][16][64]
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    *reinterpret_cast<float2*>(red + gid * kRrUnits + 8 * i + 2 * tig) = make_float2(tot[i][0], tot[i][1]);
    *reinterpret_cast<float2*>(red + (gid + 8) * kRrUnits + 8 * i + 2 * tig) = make_float2(tot[i][2], tot[i][3]);
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
  return u;
}

// A row's score but for b2, from its units j0 ... j0 + 3 (u, no bias) in each of the 16
// threads that share it.
__device__ __forceinline__ float router_row_score(const float (&u)[4], int j0, const bf16* b1, const bf16* w2) {
  float s = 0.f;
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    const float v = u[e] + __bfloat162float(b1[j0 + e]);
    s += __bfloat162float(w2[j0 + e]) * (v / (1.f + expf(-v)));
  }
  return sum16(s);
}

}  // namespace adadsf
