// Training-side pieces of AdaDSF (Sec. 3.5, Eqs. 9-11; Sec. 3.4's
// differentiable score pathway): the hidden-state alignment of one layer
// with its gradient, the output-distribution alignment (KL over the classes
// of an LM head), and the router's parameter gradient through the score gate
// of the gated variant. HBM- or latency-bound helpers around the forward;
// every reduction runs in a fixed order (results are bit-reproducible).
#include <math.h>

#include "common.cuh"
#include "internal.h"
#include "router_rows.cuh"

namespace adadsf {
namespace {

constexpr int kRowThreadsT = 256;   // 8 warps, one row per warp step
constexpr int kMaxRowBlocks = 2048;

int row_blocks(int64_t n) {
  const int64_t want = (n + 7) / 8;
  return (int)(want < kMaxRowBlocks ? (want > 0 ? want : 1) : kMaxRowBlocks);
}

// Fixed-order sum of one double per block, added to acc[0]; acc[1] += count.
__global__ void sum_partials_kernel(const double* partials, int nblocks, int64_t count, double* acc) {
  pdl_wait();
  pdl_trigger();
  __shared__ double red[256];
  double s = 0;
  for (int i = threadIdx.x; i < nblocks; i += 256) s += partials[i];
  red[threadIdx.x] = s;
  __syncthreads();
  for (int o = 128; o > 0; o >>= 1) {
    if (threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    acc[0] += red[0];
    acc[1] += (double)count;
  }
}

// Per-block fixed-order sum of the warps' per-row values.
template <int THREADS = kRowThreadsT>
__device__ __forceinline__ void block_partial(double mine, double* partials) {
  __shared__ double red[THREADS / 32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  if (lane == 0) red[w] = mine;
  __syncthreads();
  if (threadIdx.x == 0) {
    double s = 0;
    for (int i = 0; i < THREADS / 32; ++i) s += red[i];
    partials[blockIdx.x] = s;
  }
}

// Eq. 9 per row (one warp): n = |softmax(hs) - softmax(hd)| over the d
// features, and, with grad, d n / d hs = p (r / n - p . r / n) (0 if n = 0),
// p = softmax(hs), r = p - softmax(hd). fp32, four passes over the rows: the
// general path, for any d and alignment (align_hidden_vec_kernel otherwise).
template <typename T>
__global__ void __launch_bounds__(kRowThreadsT)
    align_hidden_kernel(const T* hs, const T* hd, int64_t n_rows, int d, float* grad, double* partials) {
  pdl_wait();
  pdl_trigger();
  const int lane = threadIdx.x & 31;
  const int64_t nw = (int64_t)gridDim.x * (kRowThreadsT / 32);
  double mine = 0;
  for (int64_t r = (int64_t)blockIdx.x * (kRowThreadsT / 32) + (threadIdx.x >> 5); r < n_rows; r += nw) {
    const T* a = hs + r * d;
    const T* b = hd + r * d;
    float ma = -INFINITY, mb = -INFINITY;
    for (int k = lane; k < d; k += 32) {
      ma = fmaxf(ma, Elem<T>::to_f(a[k]));
      mb = fmaxf(mb, Elem<T>::to_f(b[k]));
    }
    for (int o = 16; o > 0; o >>= 1) {
      ma = fmaxf(ma, __shfl_xor_sync(0xffffffffu, ma, o));
      mb = fmaxf(mb, __shfl_xor_sync(0xffffffffu, mb, o));
    }
    float za = 0.f, zb = 0.f;
    for (int k = lane; k < d; k += 32) {
      za += expf(Elem<T>::to_f(a[k]) - ma);
      zb += expf(Elem<T>::to_f(b[k]) - mb);
    }
    za = warp_sum(za);
    zb = warp_sum(zb);
    const float ia = 1.f / za, ib = 1.f / zb;
    float n2 = 0.f, pr = 0.f;
    for (int k = lane; k < d; k += 32) {
      const float p = expf(Elem<T>::to_f(a[k]) - ma) * ia;
      const float rr = p - expf(Elem<T>::to_f(b[k]) - mb) * ib;
      n2 = fmaf(rr, rr, n2);
      pr = fmaf(p, rr, pr);
    }
    n2 = warp_sum(n2);
    pr = warp_sum(pr);
    const float n = sqrtf(n2);
    mine += (double)n;   // identical on every lane; lane 0's copy is summed
    if (grad) {
      const float in = n > 0.f ? 1.f / n : 0.f;
      for (int k = lane; k < d; k += 32) {
        const float p = expf(Elem<T>::to_f(a[k]) - ma) * ia;
        const float rr = p - expf(Elem<T>::to_f(b[k]) - mb) * ib;
        grad[r * d + k] = p * (rr - pr) * in;
      }
    }
  }
  block_partial(mine, partials);
}

// The same with rows held in registers: 128 threads a row (one warp for rows of
// at most two 16-byte vectors a lane), NV vectors of each input a thread, loaded
// once, and each element's two exponentials computed once instead of three
// times. Three exchanges a row (maxima, sums, norm and projection). What bounds it
// is HBM: 2 n d values read and, with grad, n d floats written. At 4096 rows of
// 2048 (bf16) it takes 25 us with the gradient and 21 us without, the sum over blocks
// included (47 and 27 us on the general path: element-wise loads, one warp a row).
// Needs d a multiple of a vector's elements and 16-byte aligned pointers.
constexpr int kAlignThreads = 512;

template <typename T, int G, int NV>
__global__ void __launch_bounds__(kAlignThreads)
    align_hidden_vec_kernel(const T* hs, const T* hd, int64_t n_rows, int d, float* grad, double* partials) {
  pdl_wait();
  pdl_trigger();
  constexpr int V = Elem<T>::kVec, GROUPS = kAlignThreads / G, W = G / 32;
  __shared__ float2 xch[3][GROUPS][W];
  const int grp = threadIdx.x / G, gt = threadIdx.x % G;
  const int gw = gt >> 5, lane = threadIdx.x & 31;
  // a pair of values over the group's warps; each of the three slots is reused only
  // after the barriers of the other two
  auto exchange = [&](int slot, float2 v, auto op) {
    if (W == 1) return v;
    if (lane == 0) xch[slot][grp][gw] = v;
    named_bar_sync(1 + grp, G);
    v = xch[slot][grp][0];
#pragma unroll
    for (int w = 1; w < W; ++w) {
      const float2 f = xch[slot][grp][w];
      v = make_float2(op(v.x, f.x), op(v.y, f.y));
    }
    return v;
  };
  const auto fmx = [](float a, float b) { return fmaxf(a, b); };
  const auto fad = [](float a, float b) { return a + b; };
  const int64_t step = (int64_t)gridDim.x * GROUPS;
  double mine = 0;
  for (int64_t r = (int64_t)blockIdx.x * GROUPS + grp; r < n_rows; r += step) {
    const T* a = hs + r * d;
    const T* b = hd + r * d;
    float ea[NV][V], eb[NV][V];
    float ma = -INFINITY, mb = -INFINITY;
#pragma unroll
    for (int i = 0; i < NV; ++i) {
      const int k = (i * G + gt) * V;
      if (k < d) {
        load_vec(a + k, ea[i]);
        load_vec(b + k, eb[i]);
      }
    }
#pragma unroll
    for (int i = 0; i < NV; ++i)
      if ((i * G + gt) * V < d)
#pragma unroll
        for (int e = 0; e < V; ++e) {
          ma = fmaxf(ma, ea[i][e]);
          mb = fmaxf(mb, eb[i][e]);
        }
    for (int o = 16; o > 0; o >>= 1) {
      ma = fmaxf(ma, __shfl_xor_sync(0xffffffffu, ma, o));
      mb = fmaxf(mb, __shfl_xor_sync(0xffffffffu, mb, o));
    }
    const float2 m2 = exchange(0, make_float2(ma, mb), fmx);
    float za = 0.f, zb = 0.f;
#pragma unroll
    for (int i = 0; i < NV; ++i)
      if ((i * G + gt) * V < d)
#pragma unroll
        for (int e = 0; e < V; ++e) {
          ea[i][e] = expf(ea[i][e] - m2.x);
          eb[i][e] = expf(eb[i][e] - m2.y);
          za += ea[i][e];
          zb += eb[i][e];
        }
    const float2 z2 = exchange(1, make_float2(warp_sum(za), warp_sum(zb)), fad);
    const float ia = 1.f / z2.x, ib = 1.f / z2.y;
    float n2 = 0.f, pr = 0.f;
#pragma unroll
    for (int i = 0; i < NV; ++i)
      if ((i * G + gt) * V < d)
#pragma unroll
        for (int e = 0; e < V; ++e) {
          const float p = ea[i][e] * ia;
          const float rr = p - eb[i][e] * ib;
          n2 = fmaf(rr, rr, n2);
          pr = fmaf(p, rr, pr);
          ea[i][e] = p;
          eb[i][e] = rr;
        }
    const float2 s2 = exchange(2, make_float2(warp_sum(n2), warp_sum(pr)), fad);
    const float n = sqrtf(s2.x);
    if (gt == 0) mine += (double)n;
    if (grad) {
      const float in = n > 0.f ? 1.f / n : 0.f;
#pragma unroll
      for (int i = 0; i < NV; ++i) {
        const int k = (i * G + gt) * V;
        if (k < d) {
          float* g = grad + r * d + k;
#pragma unroll
          for (int e = 0; e < V; e += 4)
            *reinterpret_cast<float4*>(g + e) =
                make_float4(ea[i][e] * (eb[i][e] - s2.y) * in, ea[i][e + 1] * (eb[i][e + 1] - s2.y) * in,
                            ea[i][e + 2] * (eb[i][e + 2] - s2.y) * in, ea[i][e + 3] * (eb[i][e + 3] - s2.y) * in);
        }
      }
    }
  }
  block_partial<kAlignThreads>(mine, partials);
}

// Eq. 10 per row (one warp): KL(softmax(ld) || softmax(ls)) over n_cls
// classes, from fp32 logits (fp32 storage; bf16 folds the logits into the
// sums where they are computed, kl_tc.cu).
__global__ void __launch_bounds__(kRowThreadsT)
    kl_rows_kernel(const float* ls, const float* ld, int64_t n_rows, int n_cls, double* partials) {
  pdl_wait();
  pdl_trigger();
  const int lane = threadIdx.x & 31;
  const int64_t nw = (int64_t)gridDim.x * (kRowThreadsT / 32);
  double mine = 0;
  for (int64_t r = (int64_t)blockIdx.x * (kRowThreadsT / 32) + (threadIdx.x >> 5); r < n_rows; r += nw) {
    const float* a = ls + r * n_cls;
    const float* b = ld + r * n_cls;
    float ma = -INFINITY, mb = -INFINITY;
    for (int k = lane; k < n_cls; k += 32) {
      ma = fmaxf(ma, a[k]);
      mb = fmaxf(mb, b[k]);
    }
    for (int o = 16; o > 0; o >>= 1) {
      ma = fmaxf(ma, __shfl_xor_sync(0xffffffffu, ma, o));
      mb = fmaxf(mb, __shfl_xor_sync(0xffffffffu, mb, o));
    }
    float za = 0.f, zb = 0.f;
    for (int k = lane; k < n_cls; k += 32) {
      za += expf(a[k] - ma);
      zb += expf(b[k] - mb);
    }
    za = warp_sum(za);
    zb = warp_sum(zb);
    // log P = logit - max - log Z
    const float la = ma + logf(za), lb = mb + logf(zb);
    float kl = 0.f;
    for (int k = lane; k < n_cls; k += 32) {
      const float lpb = b[k] - lb;
      kl = fmaf(expf(lpb), lpb - (a[k] - la), kl);
    }
    mine += (double)warp_sum(kl);
  }
  block_partial(mine, partials);
}

// Router gradient, part 1 (16 kept rows a block; m-th kept row = flat row
// rows[m]): u = W1 x_r + b1 (h <= 64 hidden units, router_rows.cuh), s = w2 .
// SiLU(u) + b2, the gate's ds = sigmoid'(s) (G_r . delta_r) with delta_r =
// y_plain_r - x_r, and du = ds w2 SiLU'(u). Writes du [m][h], SiLU(u) [m][h]
// and ds [m]. bf16 (h = 64): u on warp-level tensor products, so the rows of x,
// y_plain and G bound it; fp32: on FFMA. G may be 4-byte aligned only (vec: 16-byte
// loads).
template <typename T>
__global__ void __launch_bounds__(kRrThreads, 2)
    router_bwd_rows_kernel(const T* x, const T* y_plain, const int32_t* rows, int64_t M, int d, int h,
                           const T* w1, const T* b1, const T* w2, const T* b2, const float* G, int vec, float* du,
                           float* su, float* ds_out) {
  pdl_wait();
  pdl_trigger();
  extern __shared__ __align__(16) float smem_rr[];
  __shared__ float gd_s[kRrRows];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t m0 = (int64_t)blockIdx.x * kRrRows;
  // G_r . delta_r: two rows a warp, 4 consecutive features a lane
  for (int i = 0; i < kRrRows / kRrWarps; ++i) {
    const int64_t m = m0 + warp * (kRrRows / kRrWarps) + i;
    float gd = 0.f;
    if (m < M) {
      const int64_t r0 = (int64_t)rows[m] * d;
#pragma unroll 4
      for (int k = lane * 4; k < d; k += 128) {
        float g[4], a[4], b[4];
        if (vec) {
          const float4 f = *reinterpret_cast<const float4*>(G + r0 + k);
          g[0] = f.x; g[1] = f.y; g[2] = f.z; g[3] = f.w;
        } else {
#pragma unroll
          for (int e = 0; e < 4; ++e) g[e] = G[r0 + k + e];
        }
        load4(x + r0 + k, a);
        load4(y_plain + r0 + k, b);
#pragma unroll
        for (int e = 0; e < 4; ++e) gd = fmaf(g[e], b[e] - a[e], gd);
      }
    }
    gd = warp_sum(gd);
    if (lane == 0) gd_s[warp * (kRrRows / kRrWarps) + i] = gd;
  }
  const int64_t ma = m0 + (lane >> 2) < M ? m0 + (lane >> 2) : M - 1;
  const int64_t mb = m0 + (lane >> 2) + 8 < M ? m0 + (lane >> 2) + 8 : M - 1;
  // its barriers make gd_s visible
  float4 u4;
  if constexpr (sizeof(T) == 2) {
    RouterPiece first;
    if (warp < d / 32) first.load_w(w1, d, warp);
    u4 = router_rows_partial(x + (int64_t)rows[ma] * d, x + (int64_t)rows[mb] * d, w1, d, 0, d / 32, first, smem_rr);
  } else {
    u4 = router_rows_units<T>(x + (int64_t)rows[ma] * d, x + (int64_t)rows[mb] * d, w1, 0, h, d, smem_rr);
  }
  const int row = threadIdx.x >> 4, j0 = (threadIdx.x & 15) * 4;
  const float uu[4] = {u4.x, u4.y, u4.z, u4.w};
  float si[4], dsi[4], s = 0.f;
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    si[e] = dsi[e] = 0.f;
    if (j0 + e < h) {
      const float u = uu[e] + Elem<T>::to_f(b1[j0 + e]);
      const float sg = 1.f / (1.f + expf(-u));
      const float wj = Elem<T>::to_f(w2[j0 + e]);
      si[e] = u * sg;
      s += wj * u * sg;
      dsi[e] = sg * (1.f + u * (1.f - sg)) * wj;   // w2 SiLU'(u), scaled by ds below
    }
  }
  s = sum16(s) + Elem<T>::to_f(b2[0]);
  const float sig = 1.f / (1.f + expf(-s));
  const float ds = sig * (1.f - sig) * gd_s[row];
  const int64_t m = m0 + row;
  if (m >= M) return;
#pragma unroll
  for (int e = 0; e < 4; ++e)
    if (j0 + e < h) {
      su[m * h + j0 + e] = si[e];
      du[m * h + j0 + e] = dsi[e] * ds;
    }
  if (j0 == 0) ds_out[m] = ds;
}

// f as a sum of three bf16 values (in the high halves of p): exact for finite f
// (each part takes the next 8 significant bits), f itself rounded where it is not.
__device__ __forceinline__ void bf16_parts(float f, uint32_t (&p)[3]) {
  const bool finite = fabsf(f) <= 3.402823466e38f;
  p[0] = finite ? __float_as_uint(f) & 0xffff0000u : (uint32_t)__bfloat16_as_ushort(__float2bfloat16_rn(f)) << 16;
  const float r = f - __uint_as_float(p[0]);
  p[1] = finite ? __float_as_uint(r) & 0xffff0000u : 0u;
  p[2] = finite ? __float_as_uint(r - __uint_as_float(p[1])) & 0xffff0000u : 0u;
}

// Router gradient, part 2: dW1[j][k] = sum_m du[m][j] x[rows[m]][k]. A cluster
// of 8 CTAs owns 64 columns k and all h <= 64 units; each CTA sums an eighth
// of the rows (rows staged 32 at a time with the next 32 in flight) and the
// eighths are added in rank order through distributed shared memory. The split
// along m is what fills the GPU: the output has only d / 64 such tiles (32 at d =
// 2048). fp32 x: 8 units x 4 columns a thread on FFMA. bf16 x: tensor products with
// du cut into three bf16 parts that add up to it exactly (8 of its 24 bits each), the
// smallest first, each 16 rows summed from zero and added in fp32, so nothing of
// du's precision is lost. The last cluster sums db1[j] = sum_m du[m][j], dw2[j] = sum_m
// ds[m] SiLU(u)[m][j] and db2 = sum_m ds[m] the same way. With part 1 it takes
// 29 us at M = 2048, d = 2048 (bf16) and 0.42 ms at M = 32768; 76 us and 0.97
// ms with both parts on FFMA, 1024 us and 20.8 ms for one warp a row with 64 serial
// dots and a reduction of 17 blocks that summed the vectors in one thread each.
constexpr int kRedCluster = 8;
constexpr int kRedThreads = 128;
constexpr int kRedCols = 64;
constexpr int kRedRows = 32;   // rows a stage

template <typename T>
__global__ void __launch_bounds__(kRedThreads)
    router_bwd_reduce_kernel(const T* x, const int32_t* rows, int64_t M, int d, int h, const float* du,
                             const float* su, const float* ds, float* grad) {
  pdl_wait();
  pdl_trigger();
  constexpr int V = Elem<T>::kVec;
  constexpr int XV = kRedRows * kRedCols / V / kRedThreads;   // 16-byte x vectors a thread
  constexpr bool MMA = sizeof(T) == 2;
  __shared__ __align__(16) float sdu[MMA ? 1 : kRedRows][64];
  __shared__ __align__(16) float sx[MMA ? 1 : kRedRows][kRedCols];
  // MMA: rows of 64 bf16, 16-byte chunks XOR-ed with row % 8; three parts of du, x
  __shared__ __align__(16) uint8_t sb[MMA ? 4 : 1][MMA ? kRedRows * 128 : 16];
  __shared__ __align__(16) float part[64 * kRedCols];
  const int rank = (int)cluster_ctarank();
  const int col0 = (int)(blockIdx.x / kRedCluster) * kRedCols;
  const int64_t m_lo = M * rank / kRedCluster, m_hi = M * (rank + 1) / kRedCluster;
  const int tid = threadIdx.x;
  if (col0 >= d) {
    // the vector sums: units over 64 threads, the rows' two halves over the block
    const int j = tid & 63, half = tid >> 6;
    float gb1 = 0.f, gw2 = 0.f, gb2 = 0.f;
    if (j < h) {
#pragma unroll 4
      for (int64_t m = m_lo + half; m < m_hi; m += 2) {
        gb1 += du[m * h + j];
        gw2 = fmaf(ds[m], su[m * h + j], gw2);
      }
    }
    for (int64_t m = m_lo + tid; m < m_hi; m += kRedThreads) gb2 += ds[m];
    gb2 = warp_sum(gb2);
    part[half * 128 + j] = gb1;
    part[half * 128 + 64 + j] = gw2;
    if ((tid & 31) == 0) part[256 + (tid >> 5)] = gb2;
    cluster_sync();
    if (rank == 0) {
      const uint32_t base = smem_u32(part);
      float a = 0.f, b = 0.f;   // thread t < 128: value t of both halves
      for (int q = 0; q < kRedCluster; ++q) {
        const uint32_t p = map_to_cta(base, q);
        a += ld_cluster_f32(p + 4 * tid) + ld_cluster_f32(p + 4 * (128 + tid));
        if (tid == 0)
          for (int w = 0; w < kRedThreads / 32; ++w) b += ld_cluster_f32(p + 4 * (256 + w));
      }
      if (j < h) grad[(int64_t)h * d + (tid >> 6) * h + j] = a;
      if (tid == 0) grad[(int64_t)h * d + 2 * h] = b;
    }
    cluster_sync();   // the partials stay until every CTA has read them
    return;
  }
  const int ty = tid >> 4, tx = tid & 15;   // FFMA: units 8 ty .. + 7, columns 4 tx .. + 3
  if constexpr (MMA) {
    const int lane = tid & 31, warp = tid >> 5;
    const int u0 = (warp >> 1) * 32, c0 = (warp & 1) * 32;   // the warp's 32 units x 32 columns
    float tot[2][4][4];
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) tot[i][j][0] = tot[i][j][1] = tot[i][j][2] = tot[i][j][3] = 0.f;
    float2 dv[kRedRows / 4];
    uint4 xv[2];
    auto fetch = [&](int64_t m0) {
#pragma unroll
      for (int i = 0; i < kRedRows / 4; ++i) {   // rows warp + 4 i, units 2 lane and + 1
        const int64_t m = m0 + warp + 4 * i;
        dv[i] = m < m_hi ? *reinterpret_cast<const float2*>(du + m * h + 2 * lane) : make_float2(0.f, 0.f);
      }
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        const int64_t m = m0 + (tid >> 3) + 16 * i;
        xv[i] = m < m_hi ? *reinterpret_cast<const uint4*>(x + (int64_t)rows[m] * d + col0 + (tid & 7) * 8)
                         : make_uint4(0, 0, 0, 0);
      }
    };
    const uint32_t sbase = smem_u32(&sb[0][0]);
    constexpr uint32_t PLANE = kRedRows * 128;
    if (m_lo < m_hi) fetch(m_lo);
    for (int64_t m0 = m_lo; m0 < m_hi; m0 += kRedRows) {
      __syncthreads();
#pragma unroll
      for (int i = 0; i < kRedRows / 4; ++i) {
        const int r = warp + 4 * i;
        uint32_t p0[3], p1[3];
        bf16_parts(dv[i].x, p0);
        bf16_parts(dv[i].y, p1);
        const uint32_t off = r * 128 + ((((uint32_t)lane >> 2) ^ (r & 7)) << 4) + (lane & 3) * 4;
#pragma unroll
        for (int k = 0; k < 3; ++k) *reinterpret_cast<uint32_t*>(&sb[k][off]) = (p0[k] >> 16) | (p1[k] & 0xffff0000u);
      }
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        const int r = (tid >> 3) + 16 * i;
        *reinterpret_cast<uint4*>(&sb[3][r * 128 + (((tid & 7) ^ (r & 7)) << 4)]) = xv[i];
      }
      __syncthreads();
      if (m0 + kRedRows < m_hi) fetch(m0 + kRedRows);
      const int mi = lane >> 3, mr = lane & 7;   // ldmatrix: this lane's matrix and row
#pragma unroll
      for (int ks = 0; ks < kRedRows; ks += 16) {
        uint32_t b[2][4];
#pragma unroll
        for (int q = 0; q < 2; ++q) {   // columns c0 + 16 q: rows ks + 8 (mi & 1), column chunk mi / 2
          const int r = ks + (mi & 1) * 8 + mr, c = (c0 >> 3) + 2 * q + (mi >> 1);
          ldmatrix_x4_trans(sbase + 3 * PLANE + r * 128 + ((c ^ (r & 7)) << 4), b[q]);
        }
#pragma unroll
        for (int mt = 0; mt < 2; ++mt) {
          uint32_t a[3][4];
          const int r = ks + (mi >> 1) * 8 + mr, c = (u0 >> 3) + 2 * mt + (mi & 1);
#pragma unroll
          for (int k = 0; k < 3; ++k) ldmatrix_x4_trans(sbase + k * PLANE + r * 128 + ((c ^ (r & 7)) << 4), a[k]);
#pragma unroll
          for (int nt = 0; nt < 4; ++nt) {
            float p[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
            for (int k = 2; k >= 0; --k)
              mma_16816(p, a[k][0], a[k][1], a[k][2], a[k][3], b[nt >> 1][(nt & 1) * 2], b[nt >> 1][(nt & 1) * 2 + 1]);
#pragma unroll
            for (int e = 0; e < 4; ++e) tot[mt][nt][e] += p[e];
          }
        }
      }
    }
    const int gid = lane >> 2, tig = lane & 3;
#pragma unroll
    for (int mt = 0; mt < 2; ++mt)
#pragma unroll
      for (int nt = 0; nt < 4; ++nt) {
        float* q = part + (u0 + 16 * mt + gid) * kRedCols + c0 + 8 * nt + 2 * tig;
        *reinterpret_cast<float2*>(q) = make_float2(tot[mt][nt][0], tot[mt][nt][1]);
        *reinterpret_cast<float2*>(q + 8 * kRedCols) = make_float2(tot[mt][nt][2], tot[mt][nt][3]);
      }
  } else {
    float acc[8][4];
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
      for (int c = 0; c < 4; ++c) acc[i][c] = 0.f;
    float dv[kRedRows * 64 / kRedThreads];
    uint4 xv[XV];
    auto fetch = [&](int64_t m0) {
#pragma unroll
      for (int i = 0; i < kRedRows * 64 / kRedThreads; ++i) {
        const int mm = i * (kRedThreads / 64) + (tid >> 6), jj = tid & 63;
        dv[i] = (m0 + mm < m_hi && jj < h) ? du[(m0 + mm) * h + jj] : 0.f;
      }
#pragma unroll
      for (int i = 0; i < XV; ++i) {
        const int v = i * kRedThreads + tid;
        const int64_t m = m0 + v / (kRedCols / V);
        xv[i] = m < m_hi ? *reinterpret_cast<const uint4*>(x + (int64_t)rows[m] * d + col0 + (v % (kRedCols / V)) * V)
                         : make_uint4(0, 0, 0, 0);
      }
    };
    if (m_lo < m_hi) fetch(m_lo);
    for (int64_t m0 = m_lo; m0 < m_hi; m0 += kRedRows) {
      __syncthreads();
#pragma unroll
      for (int i = 0; i < kRedRows * 64 / kRedThreads; ++i) sdu[i * (kRedThreads / 64) + (tid >> 6)][tid & 63] = dv[i];
#pragma unroll
      for (int i = 0; i < XV; ++i) {
        const int v = i * kRedThreads + tid;
        float f[V];
        unpack16(xv[i], f, T());
        float* p = &sx[v / (kRedCols / V)][(v % (kRedCols / V)) * V];
#pragma unroll
        for (int e = 0; e < V; e += 4) *reinterpret_cast<float4*>(p + e) = make_float4(f[e], f[e + 1], f[e + 2], f[e + 3]);
      }
      __syncthreads();
      if (m0 + kRedRows < m_hi) fetch(m0 + kRedRows);
      const int nm = (int)(m_hi - m0 < kRedRows ? m_hi - m0 : kRedRows);
#pragma unroll 4
      for (int mm = 0; mm < nm; ++mm) {
        const float4 a0 = *reinterpret_cast<const float4*>(&sdu[mm][8 * ty]);
        const float4 a1 = *reinterpret_cast<const float4*>(&sdu[mm][8 * ty + 4]);
        const float4 b = *reinterpret_cast<const float4*>(&sx[mm][4 * tx]);
        const float af[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
        const float bf[4] = {b.x, b.y, b.z, b.w};
#pragma unroll
        for (int i = 0; i < 8; ++i)
#pragma unroll
          for (int c = 0; c < 4; ++c) acc[i][c] = fmaf(af[i], bf[c], acc[i][c]);
      }
    }
#pragma unroll
    for (int i = 0; i < 8; ++i)
      *reinterpret_cast<float4*>(part + (8 * ty + i) * kRedCols + 4 * tx) =
          make_float4(acc[i][0], acc[i][1], acc[i][2], acc[i][3]);
  }
  cluster_sync();
  {
    // this CTA finishes units [8 rank, 8 rank + 8): one 16-byte piece a thread
    const int j = 8 * rank + (tid >> 4);
    const uint32_t off = smem_u32(part) + 4u * (j * kRedCols + 4 * tx);
    float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int q = 0; q < kRedCluster; ++q) {
      const float4 f = ld_cluster_f32x4(map_to_cta(off, q));
      s.x += f.x;
      s.y += f.y;
      s.z += f.z;
      s.w += f.w;
    }
    if (j < h) *reinterpret_cast<float4*>(grad + (int64_t)j * d + col0 + 4 * tx) = s;
  }
  cluster_sync();   // the partials stay until every CTA has read them
}

template <typename T>
cudaError_t router_backward_t(const void* x, const void* y_plain, const int32_t* rows, int64_t M, int d, int h,
                              const void* w1, const void* b1, const void* w2, const void* b2, const float* G, float* du,
                              float* su, float* ds, float* grad, const Dev& dev) {
  const int64_t nb = (M + kRrRows - 1) / kRrRows;
  if (nb > INT32_MAX) return cudaErrorInvalidValue;
  constexpr int smem = sizeof(T) == 2 ? RouterRows<T>::MMA_BYTES : RouterRows<T>::SMEM_BYTES;
  cudaError_t e = allow_smem<router_bwd_rows_kernel<T>, smem>();
  if (e != cudaSuccess) return e;
  const int vec = (reinterpret_cast<uintptr_t>(G) & 15u) == 0 ? 1 : 0;
  e = launch_pdl(router_bwd_rows_kernel<T>, dim3((unsigned)nb), dim3(kRrThreads), smem, dev.stream,
                 static_cast<const T*>(x), static_cast<const T*>(y_plain), rows, M, d, h, static_cast<const T*>(w1),
                 static_cast<const T*>(b1), static_cast<const T*>(w2), static_cast<const T*>(b2), G, vec, du, su, ds);
  if (e != cudaSuccess) return e;
  const unsigned ncol = (unsigned)((d + kRedCols - 1) / kRedCols) + 1;
  return launch_pdl_cluster(router_bwd_reduce_kernel<T>, dim3(ncol * kRedCluster), dim3(kRedThreads), 0, dev.stream,
                            kRedCluster, static_cast<const T*>(x), rows, M, d, h, (const float*)du, (const float*)su,
                            (const float*)ds, grad);
}

// Rows in registers where a row is whole 16-byte vectors of aligned memory, fits
// (one warp up to 2 vectors a lane, else 128 threads up to 4) and gives at least
// half of a warp's lanes a vector; the general kernel otherwise (100,000 rows
// of 64 without gradient: 41.8 us there, 43.6 us with 8 lanes of 32 at work).
template <typename T>
cudaError_t align_hidden_t(const T* hs, const T* hd, int64_t n_rows, int d, float* grad, double* partials, int nb,
                           const Dev& dev) {
  constexpr int V = Elem<T>::kVec;
  const bool vec = d % V == 0 && d / V >= 16 && ((reinterpret_cast<uintptr_t>(hs) | reinterpret_cast<uintptr_t>(hd) |
                                   reinterpret_cast<uintptr_t>(grad)) & 15u) == 0;
  const int nv32 = (d / V + 31) / 32, nv128 = (d / V + 127) / 128;
  const dim3 g((unsigned)nb), b(kAlignThreads);
  if (vec && nv32 == 1)
    return launch_pdl(align_hidden_vec_kernel<T, 32, 1>, g, b, 0, dev.stream, hs, hd, n_rows, d, grad, partials);
  if (vec && nv32 == 2)
    return launch_pdl(align_hidden_vec_kernel<T, 32, 2>, g, b, 0, dev.stream, hs, hd, n_rows, d, grad, partials);
  if (vec && nv128 == 1)
    return launch_pdl(align_hidden_vec_kernel<T, 128, 1>, g, b, 0, dev.stream, hs, hd, n_rows, d, grad, partials);
  if (vec && nv128 == 2)
    return launch_pdl(align_hidden_vec_kernel<T, 128, 2>, g, b, 0, dev.stream, hs, hd, n_rows, d, grad, partials);
  if (vec && nv128 <= 4)
    return launch_pdl(align_hidden_vec_kernel<T, 128, 4>, g, b, 0, dev.stream, hs, hd, n_rows, d, grad, partials);
  return launch_pdl(align_hidden_kernel<T>, g, dim3(kRowThreadsT), 0, dev.stream, hs, hd, n_rows, d, grad, partials);
}

}  // namespace

int train_row_blocks(int64_t n) { return row_blocks(n); }

cudaError_t sum_partials(const double* partials, int nblocks, int64_t count, double* acc, const Dev& dev) {
  return launch_pdl(sum_partials_kernel, dim3(1), dim3(256), 0, dev.stream, partials, nblocks, count, acc);
}

cudaError_t align_hidden(int dtype, const void* hs, const void* hd, int64_t n_rows, int d, float* grad,
                         double* partials, double* acc, const Dev& dev) {
  if (n_rows <= 0) return cudaSuccess;
  const int nb = row_blocks(n_rows);
  const cudaError_t e = dtype == kBF16
                            ? align_hidden_t(static_cast<const bf16*>(hs), static_cast<const bf16*>(hd), n_rows, d, grad,
                                             partials, nb, dev)
                            : align_hidden_t(static_cast<const float*>(hs), static_cast<const float*>(hd), n_rows, d,
                                             grad, partials, nb, dev);
  if (e != cudaSuccess) return e;
  return sum_partials(partials, nb, n_rows, acc, dev);
}

cudaError_t kl_rows(const float* ls, const float* ld, int64_t n_rows, int n_cls, double* partials, double* acc,
                    const Dev& dev) {
  if (n_rows <= 0) return cudaSuccess;
  const int nb = row_blocks(n_rows);
  cudaError_t e = launch_pdl(kl_rows_kernel, dim3(nb), dim3(kRowThreadsT), 0, dev.stream, ls, ld, n_rows, n_cls,
                             partials);
  if (e != cudaSuccess) return e;
  return sum_partials(partials, nb, n_rows, acc, dev);
}

cudaError_t router_backward(int dtype, const void* x, const void* y_plain, const int32_t* rows, int64_t M, int d,
                            int h, const void* w1, const void* b1, const void* w2, const void* b2, const float* G,
                            float* du, float* su, float* ds, float* grad, const Dev& dev) {
  if (h > 64) return cudaErrorInvalidValue;
  if (M <= 0) return cudaMemsetAsync(grad, 0, sizeof(float) * ((size_t)h * d + 2 * h + 1), dev.stream);
  if (dtype == kBF16)
    return router_backward_t<bf16>(x, y_plain, rows, M, d, h, w1, b1, w2, b2, G, du, su, ds, grad, dev);
  return router_backward_t<float>(x, y_plain, rows, M, d, h, w1, b1, w2, b2, G, du, su, ds, grad, dev);
}

}  // namespace adadsf
