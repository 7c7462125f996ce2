// bf16 projections of at most 16 rows (a decode step): out = epi(A . W^T).
//
// Such a product reads its weights once for a handful of multiply-adds, so what
// bounds it is how soon and how evenly the weights stream. The tensor-core kernels
// of gemm_tcgen05.cu start late for that (barriers, TMEM, one tile per CTA of 64 to
// 128 weight rows, partial tiles exchanged between the CTAs of a split): a few MB of
// weights took 8 to 15 us. Here a block takes 8-row groups of W, as evenly as the
// groups divide, its 16 warps every sixteenth 64-byte piece of K, and the first pieces
// are on their way before the block waits for the previous kernel (behind a launch of
// the same call, so that the weights do not depend on it; the first launch of a call
// waits before it reads them, 0.4 to 0.8 us more in a row of products). The product is
// warp-level (mma.sync m16n8k16): 16 weight rows are the A operand, the rows of A the
// B operand's columns. Both come straight from memory: a lane loads 16 consecutive bytes of a row, and since the order of k inside
// a product is free as long as both operands agree, those bytes are the fragment as
// they come. The warps' sums are added in warp order through shared memory
// (bit-reproducible), and the next tile's first pieces load meanwhile.
//
// Its line lies at the weights' size (MB), 28 up to 8 rows and 16 above: larger
// weights stream faster by TMA, whose boxes keep more in flight than 16 loads a lane (the second
// kernel below, or the tensor-core kernels). us per product from a cold L2, weights
// requested ahead, tensor-core kernels / here:
//   N x K            MB     1 row          16 rows
//   768 x 768        1.2    5.3 / 2.1      5.1 / 2.9
//   2304 x 768       3.5    5.4 / 2.5      5.4 / 3.2
//   768 x 3072       4.7    7.3 / 3.6      7.3 / 5.0
//   2048 x 2048      8.4    6.7 / 3.4      6.7 / 4.5
//   3584 x 3584      25.7   9.5 / 9.1      9.5 / 11.1
//   1536 x 8960      27.5   13.3 / 9.2     13.3 / 12.5
//   8192 x 2048      33.6   9.7 / 11.6     9.9 / 13.8
//   18944 x 3584     136    26.3 / 34.6    28.1 / 42.8
#include <math.h>

#include <algorithm>

#include "common.cuh"
#include "internal.h"

namespace adadsf {
namespace {

constexpr int kGrThreads = 512;
constexpr int kGrWarps = kGrThreads / 32;
constexpr int kGrU = 4;               // pieces of K a warp has in flight
constexpr int kGrMaxRows = 16;

struct RowsDev {
  const bf16* x; int64_t ldx;         // [M][K1]
  const bf16* w; int64_t ldw;         // [N][K1]; with dual the gate weight
  const bf16* w2;                     // dual: the up weight
  const bf16* x2; int64_t ldx2;       // second K source, pieces n1 ...
  const bf16* wk2; int64_t ldwk2;
  int M, groups, n1, n;               // groups: N / 8; pieces of 32 k: first source, both
  int wait_first;                     // the weights may be the previous kernel's output
  int act;
  const bf16 *bias, *bias2;
  const bf16* add; int64_t ld_add; int add_gathered;   // residual
  const int32_t* rows; int out_mapped;
  const float* gate;
  const bf16* gbase; int64_t ld_gbase;
  bf16* out; int64_t ld_out;
};

__device__ __forceinline__ uint4 ld_w(const bf16* p) {
  uint4 v;
  asm volatile("ld.global.nc.L1::no_allocate.L2::256B.v4.u32 {%0, %1, %2, %3}, [%4];"
               : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
               : "l"(p));
  return v;
}

// Output element (row m of A, column n) from its sum (v2: the up weight's, DUAL).
template <bool DUAL>
__device__ __forceinline__ void rows_epilogue(const RowsDev& p, int m, int n, float v, float v2) {
  const int64_t arow = p.rows ? (int64_t)p.rows[m] : (int64_t)m;
  if (arow < 0) return;   // a row that bypasses the layer: nothing read or written
  if (p.bias) v += __bfloat162float(p.bias[n]) + (p.bias2 ? __bfloat162float(p.bias2[n]) : 0.f);
  if (DUAL) v = v / (1.f + expf(-v)) * v2;
  else if (p.act == ACT_GELU) v = 0.5f * v * (1.f + erff(v * 0.70710678118654752f));
  if (p.add) {
    const float r = __bfloat162float(p.add[(p.add_gathered ? arow : (int64_t)m) * p.ld_add + n]);
    if (!p.gate) {
      v += r;
    } else {
      const float g = 1.f / (1.f + expf(-p.gate[arow]));
      if (p.gbase) {
        const float b = __bfloat162float(p.gbase[arow * p.ld_gbase + n]);
        v = fmaf(g, (v + r) - b, b);
      } else {
        v = fmaf(g, v, r);
      }
    }
  }
  p.out[(p.out_mapped ? arow : (int64_t)m) * p.ld_out + n] = __float2bfloat16_rn(v);
}

// Groups [0, pa.groups) are problem a's, the rest b's (b.groups 0: none). A tile is
// two groups of one problem (rows 0-7 and 8-15 of the A operand); with DUAL one
// group, its gate rows and its up rows.
template <int NT, bool DUAL>
__global__ void __launch_bounds__(kGrThreads, 1)
    gemm_rows_kernel(const __grid_constant__ RowsDev pa, const __grid_constant__ RowsDev pb) {
  constexpr int NC = NT * 8;
  constexpr int STEP = DUAL ? 1 : 2;   // groups of a tile
  __shared__ float red[kGrWarps][16 * NC];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, gid = lane >> 2, tig = lane & 3;
  const int total = pa.groups + pb.groups;
  const int lo = (int)((int64_t)total * blockIdx.x / gridDim.x), hi = (int)((int64_t)total * (blockIdx.x + 1) / gridDim.x);

  // a tile: problem, groups [g, g + cnt) of it
  struct Tile {
    bool second;
    int g, cnt, next;
  };
  auto tile_at = [&](int t) {
    Tile r;
    r.second = t >= pa.groups;
    const int end = r.second ? total : min(hi, pa.groups);
    r.cnt = min(STEP, min(hi, end) - t);
    r.g = r.second ? t - pa.groups : t;
    r.next = t + r.cnt;
    return r;
  };
  uint4 w[kGrU][2];
  // this warp's pieces c, c + 16, ... of a tile, kGrU at a time
  auto load_weights = [&](const Tile& tl, int c0) {
    const RowsDev& p = tl.second ? pb : pa;
#pragma unroll
    for (int u = 0; u < kGrU; ++u) {
      const int c = c0 + u * kGrWarps;
      w[u][0] = w[u][1] = make_uint4(0, 0, 0, 0);
      if (c < p.n) {
        const bool s2 = c >= p.n1;
        const bf16* base = s2 ? p.wk2 : p.w;
        const int64_t ld = s2 ? p.ldwk2 : p.ldw;
        const int64_t at = (int64_t)(tl.g * 8 + gid) * ld + (s2 ? c - p.n1 : c) * 32 + tig * 8;
        w[u][0] = ld_w(base + at);
        if (DUAL) w[u][1] = ld_w(p.w2 + at);
        else if (tl.cnt > 1) w[u][1] = ld_w(base + at + 8 * ld);
      }
    }
  };
  if (pa.wait_first) pdl_wait();
  Tile cur = {};
  if (lo < hi) {
    cur = tile_at(lo);
    load_weights(cur, warp);
  }
  pdl_wait();
  for (int t = lo; t < hi;) {
    const RowsDev& p = cur.second ? pb : pa;
    float acc[NT][4];
#pragma unroll
    for (int nt = 0; nt < NT; ++nt) acc[nt][0] = acc[nt][1] = acc[nt][2] = acc[nt][3] = 0.f;
    for (int c0 = warp; c0 < p.n; c0 += kGrWarps * kGrU) {
      uint4 xv[kGrU][NT];
#pragma unroll
      for (int u = 0; u < kGrU; ++u) {
        const int c = c0 + u * kGrWarps;
#pragma unroll
        for (int nt = 0; nt < NT; ++nt) {
          const int m = gid + 8 * nt < p.M ? gid + 8 * nt : 0;   // a column past M: any row, its sums are dropped
          xv[u][nt] = make_uint4(0, 0, 0, 0);
          if (c < p.n)
            xv[u][nt] = *reinterpret_cast<const uint4*>(c < p.n1 ? p.x + m * p.ldx + c * 32 + tig * 8
                                                                 : p.x2 + m * p.ldx2 + (c - p.n1) * 32 + tig * 8);
        }
      }
      uint4 wc[kGrU][2];
#pragma unroll
      for (int u = 0; u < kGrU; ++u) {
        wc[u][0] = w[u][0];
        wc[u][1] = w[u][1];
      }
      if (c0 + kGrWarps * kGrU < p.n) load_weights(cur, c0 + kGrWarps * kGrU);
#pragma unroll
      for (int u = 0; u < kGrU; ++u)
#pragma unroll
        for (int nt = 0; nt < NT; ++nt) {
          const uint4 a = wc[u][0], b = wc[u][1], v = xv[u][nt];
          mma_16816(acc[nt], a.x, b.x, a.y, b.y, v.x, v.y);
          mma_16816(acc[nt], a.z, b.z, a.w, b.w, v.z, v.w);
        }
    }
    const Tile done = cur;
    t = cur.next;
    if (t < hi) {
      cur = tile_at(t);
      load_weights(cur, warp);
    } else {
      pdl_trigger();
    }
#pragma unroll
    for (int nt = 0; nt < NT; ++nt) {
      float* q = &red[warp][gid * NC + nt * 8 + tig * 2];
      *reinterpret_cast<float2*>(q) = make_float2(acc[nt][0], acc[nt][1]);
      *reinterpret_cast<float2*>(q + 8 * NC) = make_float2(acc[nt][2], acc[nt][3]);
    }
    __syncthreads();
    constexpr int OUT = (DUAL ? 8 : 16) * NC;
    if ((int)threadIdx.x < OUT) {
      const int r = threadIdx.x / NC, m = threadIdx.x % NC;
      float v = 0.f, v2 = 0.f;
#pragma unroll
      for (int q = 0; q < kGrWarps; ++q) {
        v += red[q][r * NC + m];
        if (DUAL) v2 += red[q][(r + 8) * NC + m];
      }
      if (m < p.M && (DUAL || r < done.cnt * 8)) rows_epilogue<DUAL>(p, m, done.g * 8 + r, v, v2);
    }
    __syncthreads();
  }
}

// ---------------------------------------------------------------- larger weights
constexpr int kGsWarps = 8;           // consumer warps; one 16-k product of a stage each
constexpr int kGsThreads = 32 * (kGsWarps + 1);
constexpr int kGsGroups = 8;          // 8-row groups of W a tile takes
constexpr int kGsBox = 2048;          // bytes of 8 rows x 128 k
constexpr int kGsMaxStages = 12;
constexpr int kGsRingBytes = 184 * 1024;
// Shared memory of a launch: alignment, the ring, the warps' sums and the peer's half.
constexpr int gs_smem(int ring, int pairs, int nt) {
  return 1024 + ring + (kGsWarps * pairs * 16 + pairs * 8) * nt * 8 * 4;
}

__device__ __forceinline__ void tma_load_3d(uint32_t dst, const void* tmap, int c0, int c1, int c2, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%2, %3, %4}], [%5];" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(tmap)), "r"(c0), "r"(c1), "r"(c2), "r"(bar)
      : "memory");
}
__device__ __forceinline__ void st_cluster_f32(uint32_t addr, float v) {
  asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(addr), "f"(v) : "memory");
}

// Past the line of the kernel above a product streams through TMA. Against the
// tensor-core kernels, whose tiles of 128 weight rows and splits of 2 or 4 fill 112 to
// 144 of the SMs, the groups divide over pairs of CTAs, each CTA half of K, so
// that every SM streams and only one partial tile passes between two CTAs. A thread
// brings stages of 128 k, one box of W (U groups of 8 rows, two blocks of 128-byte swizzled
// rows) and one of A (NT groups), 2 KB a group, into a ring of up to 12 stages and 184 KB;
// each of eight warps takes one 16-k product of a stage (mma.sync: 4 U NT of them a
// stage for all, at most 64, far from a limit). The sums
// of the warps are added in warp order, the pair's halves exchange theirs and
// each finishes half of the outputs. One box of 8 rows each instead of one a stage: 47 us
// at 3584 x 18944, TMA-issue bound, to 29. Chains of products of different weights,
// requested ahead as inside a step, us each, tensor-core kernels / here:
//   N x K            MB     1 row          8 rows         16 rows
//   512 x 28672      29.4   31.4 / 28.5    31.5 / 28.6    31.4 / 29.7
//   1024 x 16384     33.6   20.2 / 18.0    20.3 / 18.2
//   2048 x 8192      33.6   13.2 / 12.2    13.1 / 12.3    13.1 / 12.7
//   2048 x 11008     45.1   15.9 / 15.2    16.0 / 15.3    16.0 / 15.7
//   3584 x 3584      25.7                                 9.6 / 9.4
//   4608 x 3584      33.0   10.7 / 9.4     10.8 / 9.5     10.8 / 9.9
//   3584 x 18944     136    29.5 / 25.9    29.7 / 26.4    29.8 / 26.8
//   4864 x 8192      79.7   21.4 / 16.6    21.6 / 16.9    21.8 / 17.3
// 16 sequences at the Qwen2.5-7B shape, two layers, 16 steps 4241 -> 4084 us. With
// more rows than one tile of 64 a pair of SMs the exchanges and the repeated rows of A
// lose: 8192 x 2048 12.5 / 14.5, 18944 x 3584 29 / 37, which stay where they were.
// tmW2 / tmX2: the second K source.
template <int NT>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kGsThreads, 1)
    gemm_rows_stream_kernel(const __grid_constant__ CUtensorMap tmW, const __grid_constant__ CUtensorMap tmX,
                            const __grid_constant__ CUtensorMap tmW2, const __grid_constant__ CUtensorMap tmX2,
                            const __grid_constant__ RowsDev p, int U, int S, int* err,
                            unsigned long long timeout_ns) {
  constexpr int NC = NT * 8;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  __shared__ uint64_t bars[2 * kGsMaxStages + 1];
  __shared__ int abort_s;
  volatile int* abort_flag = &abort_s;
  const int pairs = (U + 1) / 2;
  const uint32_t stage_bytes = (uint32_t)(U + NT) * kGsBox;
  float* red = reinterpret_cast<float*>(smem + (size_t)S * stage_bytes);   // [warp][pair][16][NC]
  float* recv = red + kGsWarps * pairs * 16 * NC;                          // [pairs * 8 * NC]: from the peer
  const uint32_t ring = smem_u32(smem), full0 = smem_u32(bars), empty0 = full0 + 8 * kGsMaxStages,
                 rbar = empty0 + 8 * kGsMaxStages;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int rank = (int)cluster_ctarank();
  const int cl = blockIdx.x >> 1, ncl = gridDim.x >> 1;
  // this pair's groups [lo, lo + cnt), cnt <= U, and this CTA's stages [k0, k1), n1 of all from the first source
  const int lo = (int)((int64_t)p.groups * cl / ncl), cnt = (int)((int64_t)p.groups * (cl + 1) / ncl) - lo;
  const int n1 = (p.n1 + 3) / 4, n = n1 + (p.n - p.n1 + 3) / 4;
  const int k0 = rank == 0 ? 0 : n / 2, k1 = rank == 0 ? n / 2 : n;

  if (threadIdx.x == 0) {
    for (int s = 0; s < S; ++s) {
      mbar_init(full0 + 8 * s, 1);
      mbar_init(empty0 + 8 * s, kGsWarps);
    }
    mbar_init(rbar, kGsWarps);
    abort_s = 0;
    fence_barrier_init();
  }
  cluster_sync();   // the peer's arrivals find the barriers initialised

  if (warp == kGsWarps) {
    if (lane == 0) {
      tma_prefetch_desc(&tmW);
      tma_prefetch_desc(&tmX);
      int stage = 0;
      uint32_t phase = 0;
      int64_t issued = 0;
      auto load_w = [&](int k, int s) {
        const bool s2 = k >= n1;
        mbar_arrive_expect_tx(full0 + 8 * s, stage_bytes);
        tma_load_3d(ring + s * stage_bytes, s2 ? &tmW2 : &tmW, 0, lo * 8, 2 * (s2 ? k - n1 : k), full0 + 8 * s);
      };
      auto load_x = [&](int k, int s) {
        const bool s2 = k >= n1;
        tma_load_3d(ring + s * stage_bytes + U * kGsBox, s2 ? &tmX2 : &tmX, 0, 0, 2 * (s2 ? k - n1 : k), full0 + 8 * s);
      };
      // behind a launch of the same call the weights do not depend on the kernel before
      if (p.wait_first) pdl_wait();
      const int pre = min(S, k1 - k0);
      for (int i = 0; i < pre; ++i) load_w(k0 + i, i);
      pdl_wait();
      for (int k = k0; k < k1; ++k) {
        if (k - k0 >= pre) {
          if (!mbar_wait_bounded(empty0 + 8 * stage, phase ^ 1, abort_flag, err, timeout_ns)) break;
          load_w(k, stage);
        }
        load_x(k, stage);
        ++issued;
        if (++stage == S) { stage = 0; phase ^= 1; }
      }
      pdl_trigger();
      for (int s = 0; s < S && s < issued; ++s) {   // every copy has landed before the block goes
        const int64_t last = s + ((issued - 1 - s) / S) * S;
        mbar_wait_drain(full0 + 8 * s, (uint32_t)((last / S) & 1), timeout_ns);
      }
    }
    __syncwarp();
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  } else {
    pdl_wait();
    // this warp's product of a stage: 16-byte columns ck and ck + 1 of the stage's column kb
    const int kb = warp >> 2, ck = (warp & 3) * 2;
    const int wr = (lane & 7) + ((lane >> 3) & 1) * 8;   // ldmatrix row of W: two groups
    const uint32_t w_at = (uint32_t)(kb * U * 1024 + wr * 128 + (((ck + (lane >> 4)) ^ (wr & 7)) << 4));
    const int xr = (lane & 7) + (NT == 2 ? (lane >> 4) * 8 : 0);
    const uint32_t x_at = (uint32_t)(U * kGsBox + kb * 1024 * NT + xr * 128 + (((ck + ((lane >> 3) & 1)) ^ (xr & 7)) << 4));
    const int gid = lane >> 2, tig = lane & 3;
    int stage = 0;
    uint32_t phase = 0;
    bool ok = true;   // after a wait that ran out the warps go on without waiting, to the end
    float acc[kGsGroups / 2][NT][4];
#pragma unroll
    for (int q = 0; q < kGsGroups / 2; ++q)
#pragma unroll
      for (int nt = 0; nt < NT; ++nt) acc[q][nt][0] = acc[q][nt][1] = acc[q][nt][2] = acc[q][nt][3] = 0.f;
    for (int k = k0; k < k1; ++k) {
      ok = __all_sync(~0u, mbar_wait_bounded(full0 + 8 * stage, phase, abort_flag, err, timeout_ns));
      if (!ok) break;
      const uint32_t base = ring + stage * stage_bytes;
      uint32_t xv[4];
      ldmatrix_x4(base + x_at, xv);
#pragma unroll
      for (int q = 0; q < kGsGroups / 2; ++q) {
        if (2 * q < cnt) {   // with an odd count the last 8 rows are others' bytes: their sums are dropped
          uint32_t wv[4];
          ldmatrix_x4(base + q * 2 * 1024 + w_at, wv);
#pragma unroll
          for (int nt = 0; nt < NT; ++nt)
            mma_16816(acc[q][nt], wv[0], wv[1], wv[2], wv[3], xv[2 * nt], xv[2 * nt + 1]);
        }
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(empty0 + 8 * stage);
      if (++stage == S) { stage = 0; phase ^= 1; }
    }
    float* mine = red + warp * pairs * 16 * NC;
#pragma unroll
    for (int q = 0; q < kGsGroups / 2; ++q) {
      if (2 * q < cnt) {
#pragma unroll
        for (int nt = 0; nt < NT; ++nt) {
          float* d = mine + (q * 16 + gid) * NC + nt * 8 + tig * 2;
          *reinterpret_cast<float2*>(d) = make_float2(acc[q][nt][0], acc[q][nt][1]);
          *reinterpret_cast<float2*>(d + 8 * NC) = make_float2(acc[q][nt][2], acc[q][nt][3]);
        }
      }
    }
    named_bar_sync(1, kGsWarps * 32);
    // the peer's half of the outputs goes to the peer, then this CTA's half is finished
    const int half = cnt * 4 * NC;
    const uint32_t to = map_to_cta(smem_u32(recv), (uint32_t)(rank ^ 1));
    for (int o = threadIdx.x; o < half; o += kGsWarps * 32) {
      float v = 0.f;
#pragma unroll
      for (int w = 0; w < kGsWarps; ++w) v += red[w * pairs * 16 * NC + (rank ^ 1) * half + o];
      st_cluster_f32(to + 4 * o, v);
    }
    __syncwarp();
    if (lane == 0) mbar_arrive_cluster(map_to_cta(rbar, (uint32_t)(rank ^ 1)));
    if (ok) mbar_wait_bounded(rbar, 0, abort_flag, err, timeout_ns);
    asm volatile("fence.acq_rel.cluster;" ::: "memory");
    __syncwarp();
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    for (int o = threadIdx.x; o < half; o += kGsWarps * 32) {
      float v = 0.f;
#pragma unroll
      for (int w = 0; w < kGsWarps; ++w) v += red[w * pairs * 16 * NC + rank * half + o];
      const int e = rank * half + o, m = e % NC;
      if (m < p.M) rows_epilogue<false>(p, m, lo * 8 + e / NC, v + recv[o], 0.f);
    }
  }
  __syncwarp();
  // the peer has written its sums here before this CTA's memory goes
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

bool rows_dev(const GemmArgs& a, RowsDev& p) {
  p = RowsDev{};
  if (a.M <= 0 || a.M > kGrMaxRows || a.N % 8 || a.K % 32 || a.K2 % 32 || a.a_gather) return false;
  const Epilogue& e = a.epi;
  if (e.rope_tab || e.vt || e.nrm_psum || e.sq_out || e.cos_out || (e.add_packed && e.add_rows)) return false;
  if (e.gate_scores && (e.gate_base ? !e.add_packed : !e.add_rows)) return false;
  if (e.bias2 && !e.bias) return false;
  auto bp = [](const void* v) { return static_cast<const bf16*>(v); };
  p.x = bp(a.A); p.ldx = a.lda;
  p.w = bp(a.W); p.ldw = a.ldw;
  p.w2 = bp(a.W2);
  p.x2 = bp(a.A2); p.ldx2 = a.lda2;
  p.wk2 = bp(a.Wk2); p.ldwk2 = a.ldwk2;
  p.M = (int)a.M;
  p.groups = a.N / 8;
  p.n1 = a.K / 32;
  p.n = p.n1 + (a.K2 > 0 ? a.K2 / 32 : 0);
  p.act = e.act;
  p.bias = bp(e.bias);
  p.bias2 = bp(e.bias2);
  if (e.add_packed) {
    p.add = bp(e.add_packed);
    p.ld_add = e.ld_add_packed;
  } else if (e.add_rows) {
    p.add = bp(e.add_rows);
    p.ld_add = e.ld_add_rows;
    p.add_gathered = e.rows ? 1 : 0;
  }
  p.rows = e.rows;
  p.out_mapped = e.out_mapped ? 1 : 0;
  p.gate = e.gate_scores;
  p.gbase = bp(e.gate_base);
  p.ld_gbase = e.ld_gate_base;
  p.out = static_cast<bf16*>(e.out);
  p.ld_out = e.ld_out;
  return true;
}

double weight_bytes(const GemmArgs& g) {
  return 2.0 * g.N * ((double)(g.epi.act == ACT_SWIGLU ? 2 : 1) * g.K + (g.K2 > 0 ? g.K2 : 0));
}

// Weights (bytes) up to which the first kernel is the faster one.
double rows_line(const GemmArgs& a) { return a.M <= 8 ? 28e6 : 16e6; }

// Products for the streaming kernel: more weights than that, one tile a pair of CTAs (64
// columns a pair of SMs). From 512 columns on it is the faster one (512 x 28672 31.4 us by the
// tensor-core kernels, 29.7 here); below, too few pairs of CTAs have a group.
bool streams(const GemmArgs& a, int num_sms) {
  return a.epi.act != ACT_SWIGLU && a.K % 64 == 0 && a.K2 % 64 == 0 && a.N >= 512 &&
         a.N / 8 <= kGsGroups * (num_sms / 2) &&
         weight_bytes(a) > rows_line(a);
}

template <int NT>
cudaError_t launch_stream(const GemmArgs& a, const RowsDev& p, const Dev& dev) {
  const int ncl = std::min(dev.num_sms / 2, p.groups);
  const int U = (p.groups + ncl - 1) / ncl, pairs = (U + 1) / 2;
  CUtensorMap w, x, w2, x2;
  auto map = [](CUtensorMap* m, const void* ptr, int64_t rows, int k, int64_t ld, int box_rows) {
    return make_tmap_bf16_k(m, ptr, (uint64_t)rows, (uint64_t)k, (uint64_t)ld, (uint32_t)box_rows);
  };
  if (!map(&w, a.W, a.N, a.K, a.ldw, 8 * U) || !map(&x, a.A, a.M, a.K, a.lda, 8 * NT)) return cudaErrorInvalidValue;
  w2 = w;
  x2 = x;
  if (a.K2 > 0 && (!map(&w2, a.Wk2, a.N, a.K2, a.ldwk2, 8 * U) || !map(&x2, a.A2, a.M, a.K2, a.lda2, 8 * NT)))
    return cudaErrorInvalidValue;
  const int stage = (U + NT) * kGsBox, S = std::min(kGsMaxStages, kGsRingBytes / stage);
  const int smem = gs_smem(S * stage, pairs, NT);
  const cudaError_t e = allow_smem<gemm_rows_stream_kernel<NT>, gs_smem(kGsRingBytes, kGsGroups / 2, NT)>();
  if (e != cudaSuccess) return e;
  return launch_pdl(gemm_rows_stream_kernel<NT>, dim3((unsigned)(2 * ncl)), dim3(kGsThreads), (size_t)smem, dev.stream, w,
                    x, w2, x2, p, U, S, dev.err, kWaitTimeoutNs);
}

}  // namespace

bool gemm_rows_takes(const GemmArgs& a, const GemmArgs* b, int num_sms) {
  RowsDev p;
  if (!rows_dev(a, p) || (b && !rows_dev(*b, p))) return false;
  if (b && (a.epi.act == ACT_SWIGLU || b->epi.act == ACT_SWIGLU || a.M != b->M)) return false;
  return weight_bytes(a) + (b ? weight_bytes(*b) : 0.0) <= rows_line(a) || (!b && streams(a, num_sms));
}

cudaError_t gemm_rows(const GemmArgs& a, const GemmArgs* b, const Dev& dev) {
  RowsDev p, q = {};
  if (!rows_dev(a, p) || (b && !rows_dev(*b, q))) return cudaErrorInvalidValue;
  p.wait_first = dev.behind_own ? 0 : 1;
  if (!b && streams(a, dev.num_sms)) return a.M <= 8 ? launch_stream<1>(a, p, dev) : launch_stream<2>(a, p, dev);
  const dim3 grid((unsigned)std::min(dev.num_sms, p.groups + q.groups)), block(kGrThreads);
  if (a.epi.act == ACT_SWIGLU)
    return a.M <= 8 ? launch_pdl(gemm_rows_kernel<1, true>, grid, block, 0, dev.stream, p, q)
                    : launch_pdl(gemm_rows_kernel<2, true>, grid, block, 0, dev.stream, p, q);
  return a.M <= 8 ? launch_pdl(gemm_rows_kernel<1, false>, grid, block, 0, dev.stream, p, q)
                  : launch_pdl(gemm_rows_kernel<2, false>, grid, block, 0, dev.stream, p, q);
}

}  // namespace adadsf
