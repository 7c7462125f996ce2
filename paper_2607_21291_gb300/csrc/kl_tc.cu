// Eq. 10 on the 5th-generation tensor cores (bf16): the sum over rows of
// KL(softmax(hd W^T) || softmax(hs W^T)), W the LM head, without storing a logit.
//
// Two products share W: a CTA's tile is 128 rows by 128 classes of both, in two
// TMEM accumulators (tcgen05.mma, M = N = 128, fp32), and its epilogue folds the
// tile into running sums per row:
//   Zs = sum e^(ls - ms),  Zd = sum e^(ld - md),  X = sum e^(ld - md) (ld - ls)
// (ms, md the running maxima), from which KL = X / Zd + log(Zs / Zd) + ms - md.
// Storing the logits and reading them back cost more than the products: 4 bytes
// written and three times read per class, row and model (2 GB at 1000 rows of
// 50304 classes). There the whole loss took 1492 us (two projections of 123 us
// and a pass of 964 us over the logits); it takes 126 us here, bound by the rate
// at which one thread issues N = 128 products (two a 16-deep k step); W comes
// from HBM once, since the row blocks walk the classes side by side.
//
// Tiles are numbered row block major and the persistent CTAs take equal
// contiguous ranges, so a CTA stays on one row block (parts of two, or with few
// classes and many rows several whole ones) and keeps its sums in registers: one
// thread per row and half of a tile's columns. At the end of a row block's tiles it
// writes the five sums;
// kl_merge_kernel adds each row's records in a fixed order, in double.
//   warp 0     TMA: hs, hd and W tiles of 64 k, 4 stages of 48 KB
//   warp 1     TMEM, MMA issue (one thread); accumulators double-buffered
//   warps 2-9  epilogue (two per TMEM lane quarter, 64 classes each)
// Every barrier wait is bounded in time (device error word on give-up).
#include <cuda.h>

#include <algorithm>

#include "common.cuh"
#include "internal.h"

namespace adadsf {
namespace {

constexpr int kKlM = 128, kKlN = 128, kKlK = 64;
constexpr int kKlStages = 4;
constexpr int kKlTile = 128 * kKlK * 2;            // bytes of one operand tile
constexpr int kKlStage = 3 * kKlTile;              // hs, hd, W
constexpr int kKlEpiWarps = 8;
constexpr int kKlThreads = 64 + 32 * kKlEpiWarps;
constexpr int kKlBars = 2 * kKlStages + 5;
constexpr int kKlSmem = kKlStages * kKlStage + 1024 + kKlBars * 8 + 16;
constexpr int kKlRec = 5;                          // floats of a record: ms, Zs, md, Zd, X

struct KlDev {
  int M, N, K;
  int num_m, num_n;
  float* rec;   // [piece][row][half][kKlRec]
  int* err;
  unsigned long long timeout_ns;
};

// First tile of CTA c of G, and the CTA that holds tile t.
__host__ __device__ __forceinline__ int64_t kl_first(int64_t tiles, int G, int c) { return tiles * c / G; }
__host__ __device__ __forceinline__ int kl_owner(int64_t tiles, int G, int64_t t) {
  return (int)(((t + 1) * G - 1) / tiles);
}

// Running sums of a row; ms, md: its running maxima, which differences are taken
// from before they are scaled to powers of two (scaled maxima would leave their own
// rounding in the exponent, past any bound from logits near 1e9 on).
struct KlSums {
  float ms, zs, md, zd, x;
};
__device__ __forceinline__ float kl_ex2(float x) {   // ex2.approx: relative error ~2^-22, averaged out over the classes
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float2 f2(uint32_t a, uint32_t b) {
  return make_float2(__uint_as_float(a), __uint_as_float(b));
}
// One 32-class chunk folded in; paired fp32 arithmetic (an epilogue of accurate
// exponentials, 17 instructions each, took longer than the chunk's products).
__device__ __forceinline__ void kl_fold(KlSums& s, const uint32_t* us, const uint32_t* ud) {
  constexpr float kLog2e = 1.4426950408889634f;
  float cs[2] = {-INFINITY, -INFINITY}, cd[2] = {-INFINITY, -INFINITY};
#pragma unroll
  for (int i = 0; i < 32; ++i) {
    cs[i & 1] = fmaxf(cs[i & 1], __uint_as_float(us[i]));
    cd[i & 1] = fmaxf(cd[i & 1], __uint_as_float(ud[i]));
  }
  const float ns = fmaxf(cs[0], cs[1]), nd = fmaxf(cd[0], cd[1]);
  if (ns > s.ms || nd > s.md) {
    const float ms = fmaxf(s.ms, ns), md = fmaxf(s.md, nd);
    // a maximum that stays where it is (at -inf too) scales by 1; without one so far the sums are 0
    const float fs = ms == s.ms ? 1.f : kl_ex2((s.ms - ms) * kLog2e), fd = md == s.md ? 1.f : kl_ex2((s.md - md) * kLog2e);
    s.zs *= fs;
    s.zd *= fd;
    s.x *= fd;
    s.ms = ms;
    s.md = md;
  }
  // a maximum of -inf (every logit so far) subtracts nothing, so that the exponentials are 0
  const float ms = s.ms == -INFINITY ? 0.f : s.ms, md = s.md == -INFINITY ? 0.f : s.md;
  const float2 l2 = make_float2(kLog2e, kLog2e), ms2 = make_float2(-ms, -ms), md2 = make_float2(-md, -md);
  const float2 minus = make_float2(-1.f, -1.f), zero = make_float2(0.f, 0.f);
  float2 zs[2] = {zero, zero}, zd[2] = {zero, zero}, x[2] = {zero, zero};
#pragma unroll
  for (int i = 0; i < 16; ++i) {
    const float2 a = f2(us[2 * i], us[2 * i + 1]), b = f2(ud[2 * i], ud[2 * i + 1]);
    const float2 ta = __fmul2_rn(__fadd2_rn(a, ms2), l2), tb = __fmul2_rn(__fadd2_rn(b, md2), l2);
    const float2 e = make_float2(kl_ex2(tb.x), kl_ex2(tb.y));
    zs[i & 1] = __fadd2_rn(zs[i & 1], make_float2(kl_ex2(ta.x), kl_ex2(ta.y)));
    zd[i & 1] = __fadd2_rn(zd[i & 1], e);
    x[i & 1] = __ffma2_rn(e, __ffma2_rn(a, minus, b), x[i & 1]);
  }
  s.zs += (zs[0].x + zs[0].y) + (zs[1].x + zs[1].y);
  s.zd += (zd[0].x + zd[0].y) + (zd[1].x + zd[1].y);
  s.x += (x[0].x + x[0].y) + (x[1].x + x[1].y);
}

__global__ void __launch_bounds__(kKlThreads, 1)
    kl_tc_kernel(const __grid_constant__ CUtensorMap tmS, const __grid_constant__ CUtensorMap tmD,
                 const __grid_constant__ CUtensorMap tmW, const KlDev p) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                             ~static_cast<uintptr_t>(1023));
  const uint32_t ring = smem_u32(smem);
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + kKlStages * kKlStage);
  const uint32_t full0 = smem_u32(bars);
  const uint32_t empty0 = full0 + 8 * kKlStages;
  const uint32_t tfull0 = empty0 + 8 * kKlStages;
  const uint32_t tempty0 = tfull0 + 16;
  const uint32_t drain = tempty0 + 16;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + kKlBars);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;
  const int64_t tiles = (int64_t)p.num_m * p.num_n;
  const int64_t t0 = kl_first(tiles, gridDim.x, blockIdx.x), t1 = kl_first(tiles, gridDim.x, blockIdx.x + 1);
  const int nkb = (p.K + kKlK - 1) / kKlK;

  if (threadIdx.x == 0) {
    for (int s = 0; s < kKlStages; ++s) {
      mbar_init(full0 + 8 * s, 1);
      mbar_init(empty0 + 8 * s, 1);
    }
    for (int a = 0; a < 2; ++a) {
      mbar_init(tfull0 + 8 * a, 1);
      mbar_init(tempty0 + 8 * a, kKlEpiWarps);
    }
    mbar_init(drain, 1);
    *abort_flag = 0;
    fence_barrier_init();
    fence_proxy_async_smem();
  }
  if (warp == 0 && lane == 0) {
    tma_prefetch_desc(&tmS);
    tma_prefetch_desc(&tmD);
    tma_prefetch_desc(&tmW);
  }
  if (warp == 1) tmem_alloc(smem_u32(tmem_slot), 512);
  __syncwarp();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;

  if (warp == 0) {
    // ------------------------------------------------------------ TMA producer
    if (lane == 0) {
      pdl_wait();
      int stage = 0;
      uint32_t phase = 0;
      int64_t issued = 0;
      bool ok = true;
      for (int64_t t = t0; t < t1 && ok; ++t) {
        const int mb = (int)(t / p.num_n), nb = (int)(t % p.num_n);
        for (int kb = 0; kb < nkb; ++kb) {
          if (!mbar_wait_bounded(empty0 + 8 * stage, phase ^ 1, abort_flag, p.err, p.timeout_ns)) {
            ok = false;
            break;
          }
          const uint32_t fb = full0 + 8 * stage, dst = ring + stage * kKlStage;
          mbar_arrive_expect_tx(fb, kKlStage);
          tma_load_2d(dst, &tmS, kb * kKlK, mb * kKlM, fb);
          tma_load_2d(dst + kKlTile, &tmD, kb * kKlK, mb * kKlM, fb);
          tma_load_2d(dst + 2 * kKlTile, &tmW, kb * kKlK, nb * kKlN, fb);
          ++issued;
          if (++stage == kKlStages) { stage = 0; phase ^= 1; }
        }
      }
      for (int s = 0; s < kKlStages; ++s) {   // drain: the copies issued last have landed
        if (issued <= s) break;
        const int64_t last = s + ((issued - 1 - s) / kKlStages) * kKlStages;
        mbar_wait_drain(full0 + 8 * s, (uint32_t)((last / kKlStages) & 1), p.timeout_ns);
      }
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------ MMA issuer
    if (lane == 0) {
      constexpr uint32_t idesc = idesc_bf16_f32(kKlM, kKlN);
      int stage = 0;
      uint32_t phase = 0;
      int it = 0;
      bool ok = true;
      for (int64_t t = t0; t < t1 && ok; ++t, ++it) {
        const int acc = it & 1;
        if (!mbar_wait_bounded(tempty0 + 8 * acc, ((it >> 1) & 1) ^ 1, abort_flag, p.err, p.timeout_ns)) break;
        tc_fence_after();
        const uint32_t d_s = tmem_base + acc * 256, d_d = d_s + 128;
        for (int kb = 0; kb < nkb; ++kb) {
          if (!mbar_wait_bounded(full0 + 8 * stage, phase, abort_flag, p.err, p.timeout_ns)) {
            ok = false;
            break;
          }
          tc_fence_after();
          const uint32_t src = ring + stage * kKlStage;
#pragma unroll
          for (int k = 0; k < kKlK / 16; ++k) {
            const uint64_t wd = smem_desc_sw128(src + 2 * kKlTile + k * 32);
            const uint32_t accum = (kb > 0 || k > 0) ? 1u : 0u;
            tc_mma_f16(d_s, smem_desc_sw128(src + k * 32), wd, idesc, accum);
            tc_mma_f16(d_d, smem_desc_sw128(src + kKlTile + k * 32), wd, idesc, accum);
          }
          tc_commit(empty0 + 8 * stage);
          if (++stage == kKlStages) { stage = 0; phase ^= 1; }
        }
        if (ok) tc_commit(tfull0 + 8 * acc);
      }
      tc_commit(drain);
      mbar_wait_drain(drain, 0, p.timeout_ns);
    }
  } else {
    // ------------------------------------------------------------ epilogue
    pdl_wait();   // the records may still be read by an earlier call's merge
    const int quarter = warp & 3, half = (warp - 2) >> 2;
    const int row = quarter * 32 + lane;
    const uint32_t lane_off = (uint32_t)(quarter * 32) << 16;
    KlSums s = {-INFINITY, 0.f, -INFINITY, 0.f, 0.f};
    int it = 0;
    for (int64_t t = t0; t < t1; ++t, ++it) {
      const int mb = (int)(t / p.num_n), nb = (int)(t % p.num_n);
      const int acc = it & 1;
      int ok = 0;
      if (lane == 0) ok = mbar_wait_bounded(tfull0 + 8 * acc, (it >> 1) & 1, abort_flag, p.err, p.timeout_ns);
      ok = __shfl_sync(0xffffffffu, ok, 0);
      if (!ok) break;
      tc_fence_after();
      const uint32_t ts = tmem_base + lane_off + acc * 256 + half * 64;
#pragma unroll 1
      for (int c = 0; c < 2; ++c) {
        if (nb * kKlN + half * 64 + c * 32 >= p.N) break;   // N is a multiple of 64: whole chunks
        uint32_t us[32], ud[32];
        tmem_ld32(ts + c * 32, us);
        tmem_ld32(ts + 128 + c * 32, ud);
        tmem_ld_wait();
        kl_fold(s, us, ud);
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(tempty0 + 8 * acc);
      if (t + 1 == t1 || nb + 1 == p.num_n) {
        // this CTA's share of the row block is done
        const int piece = (int)blockIdx.x - kl_owner(tiles, gridDim.x, (int64_t)mb * p.num_n);
        const int64_t m = (int64_t)mb * kKlM + row;
        if (m < p.M) {
          float* r = p.rec + (((int64_t)piece * p.M + m) * 2 + half) * kKlRec;
          r[0] = s.ms;
          r[1] = s.zs;
          r[2] = s.md;
          r[3] = s.zd;
          r[4] = s.x;
        }
        s = {-INFINITY, 0.f, -INFINITY, 0.f, 0.f};
      }
    }
  }

  __syncwarp();
  tc_fence_before();
  __syncthreads();
  // only now: the merge's small blocks, let in at the start, sat beside this
  // kernel's and slowed it by 38 us (185 -> 148 us, 1000 rows of 50304 classes)
  pdl_trigger();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem_base, 512);
  }
}

// The records of each row into its KL, L lanes a row (the other lanes of a warp take
// other rows), then one double per block, in a fixed order. A half without a class (ms =
// md = -inf, sums 0) adds nothing.
// L = 1 or 32: an instruction in fp64 takes the SM as long for one lane as for 32, so
// that a lane a row does the division and logarithm of 32 rows at once, and its walk
// along the records is no longer than a warp's sum over its lanes while there are
// few. In all, us, warp / lane a row: 40,000 rows of 64 classes (2 to 6 records) 196 / 25,
// 20,000 of 1024 135 / 49, 4096 of 50304 (up to 12) 321 / 309, 2000 of 50304 (22) 168 / 173,
// 1000 of 50304 (42) 90 / 112 (d = 512).
constexpr int kKlFewRecords = 16;

template <int L>
__global__ void __launch_bounds__(256)
    kl_merge_kernel(const float* rec, int M, int num_n, int64_t tiles, int G, double* partials) {
  pdl_wait();
  pdl_trigger();
  __shared__ double red[8];
  constexpr int ROWS = 256 / L;   // rows a block takes at once
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, li = threadIdx.x % L;
  double mine = 0.0;
  for (int64_t m = (int64_t)blockIdx.x * ROWS + threadIdx.x / L; m < M; m += (int64_t)gridDim.x * ROWS) {
    const int64_t mb = m / kKlM;
    const int n = 2 * (kl_owner(tiles, G, (mb + 1) * num_n - 1) - kl_owner(tiles, G, mb * num_n) + 1);
    auto at = [&](int i) { return rec + (((int64_t)(i >> 1) * M + m) * 2 + (i & 1)) * kKlRec; };
    float ms = -INFINITY, md = -INFINITY;
    for (int i = li; i < n; i += L) {
      ms = fmaxf(ms, at(i)[0]);
      md = fmaxf(md, at(i)[2]);
    }
    if (L == 32)
      for (int o = 16; o > 0; o >>= 1) {
        ms = fmaxf(ms, __shfl_xor_sync(0xffffffffu, ms, o));
        md = fmaxf(md, __shfl_xor_sync(0xffffffffu, md, o));
      }
    double zs = 0.0, zd = 0.0, x = 0.0;
    for (int i = li; i < n; i += L) {
      const float* r = at(i);
      const float fs = r[0] == ms ? 1.f : expf(r[0] - ms), fd = r[2] == md ? 1.f : expf(r[2] - md);
      zs += (double)r[1] * fs;
      zd += (double)r[3] * fd;
      x += (double)r[4] * fd;
    }
    if (L == 32) {
      zs = warp_sum(zs);
      zd = warp_sum(zd);
      x = warp_sum(x);
    }
    if (li == 0) mine += x / zd + log(zs / zd) + ((double)ms - (double)md);
  }
  if (L == 1) mine = warp_sum(mine);   // L == 32: lane 0 has the warp's
  if (lane == 0) red[warp] = mine;
  __syncthreads();
  if (threadIdx.x == 0) {
    double s = 0.0;
    for (int i = 0; i < 8; ++i) s += red[i];
    partials[blockIdx.x] = s;
  }
}

}  // namespace

cudaError_t kl_tc(const void* hs, const void* hd, const void* w, int64_t n_rows, int d, int n_cls, float* rec,
                  double* partials, double* acc, const Dev& dev) {
  if (n_rows <= 0) return cudaSuccess;
  if (n_rows > INT32_MAX - kKlM || n_cls % 64 || d % 64) return cudaErrorInvalidValue;
  cudaError_t e = allow_smem<kl_tc_kernel, kKlSmem>();
  if (e != cudaSuccess) return e;
  CUtensorMap ts, td, tw;
  if (!make_tmap_bf16(&ts, hs, (uint64_t)n_rows, (uint64_t)d, (uint64_t)d, kKlK, kKlM) ||
      !make_tmap_bf16(&td, hd, (uint64_t)n_rows, (uint64_t)d, (uint64_t)d, kKlK, kKlM) ||
      !make_tmap_bf16(&tw, w, (uint64_t)n_cls, (uint64_t)d, (uint64_t)d, kKlK, kKlN))
    return cudaErrorInvalidValue;
  KlDev p;
  p.M = (int)n_rows;
  p.N = n_cls;
  p.K = d;
  p.num_m = (int)((n_rows + kKlM - 1) / kKlM);
  p.num_n = (n_cls + kKlN - 1) / kKlN;
  p.rec = rec;
  p.err = dev.err;
  p.timeout_ns = kWaitTimeoutNs;
  const int64_t tiles = (int64_t)p.num_m * p.num_n;
  const int G = (int)std::min<int64_t>(tiles, dev.num_sms);
  e = launch_pdl(kl_tc_kernel, dim3((unsigned)G), dim3(kKlThreads), kKlSmem, dev.stream, ts, td, tw, p);
  if (e != cudaSuccess) return e;
  // records of a row, at most: the CTAs whose ranges a row block's tiles touch, two each
  const int64_t records = 2 * std::min<int64_t>(G, p.num_n / (tiles / G) + 2);
  const bool few = records <= kKlFewRecords;
  const int nb = few ? (int)std::min<int64_t>(train_row_blocks(n_rows), (n_rows + 255) / 256) : train_row_blocks(n_rows);
  e = few ? launch_pdl(kl_merge_kernel<1>, dim3((unsigned)nb), dim3(256), 0, dev.stream, (const float*)rec, p.M, p.num_n,
                       tiles, G, partials)
          : launch_pdl(kl_merge_kernel<32>, dim3((unsigned)nb), dim3(256), 0, dev.stream, (const float*)rec, p.M, p.num_n,
                       tiles, G, partials);
  if (e != cudaSuccess) return e;
  return sum_partials(partials, nb, n_rows, acc, dev);
}

}  // namespace adadsf
