// bf16 projections of at most 16 rows (a decode step): out = epi(A . W^T).
//
// Such a product reads its weights once for a handful of multiply-adds, so what
// bounds it is how soon and how evenly the weights stream. The tensor-core kernels
// of gemm_tcgen05.cu start late for that (barriers, TMEM, one tile per CTA of 64 to
// 128 weight rows, partial tiles exchanged between the CTAs of a split): a few MB of
// weights took 8 to 15 us. Here a block takes 8-row groups of W, as evenly as the
// groups divide, its 16 warps every sixteenth 64-byte piece of K, and the first pieces
// are on their way before the block waits for the previous kernel (weights do not
// depend on it). The product is warp-level (mma.sync m16n8k16): 16 weight rows
// are the A operand, the rows of A the B operand's columns. Both come straight from
// memory: a lane loads 16 consecutive bytes of a row, and since the order of k inside
// a product is free as long as both operands agree, those bytes are the fragment as
// they come. The warps' sums are added in warp order through shared memory
// (bit-reproducible), and the next tile's first pieces load meanwhile.
//
// The line to the tensor-core kernels lies at the weights' size (MB), 28 up to 8 rows
// and 16 above, because those stream large weights faster (TMA boxes keep more in
// flight than 16 loads a lane). us per product from a cold L2, there / here:
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

__device__ __forceinline__ void mma_rows(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0,
                                         uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, "
      "{%8, %9}, {%0, %1, %2, %3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
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
          mma_rows(acc[nt], a.x, b.x, a.y, b.y, v.x, v.y);
          mma_rows(acc[nt], a.z, b.z, a.w, b.w, v.z, v.w);
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

}  // namespace

bool gemm_rows_takes(const GemmArgs& a, const GemmArgs* b) {
  RowsDev p;
  if (!rows_dev(a, p) || (b && !rows_dev(*b, p))) return false;
  if (b && (a.epi.act == ACT_SWIGLU || b->epi.act == ACT_SWIGLU || a.M != b->M)) return false;
  auto bytes = [](const GemmArgs& g) {
    return 2.0 * g.N * ((double)(g.epi.act == ACT_SWIGLU ? 2 : 1) * g.K + (g.K2 > 0 ? g.K2 : 0));
  };
  return bytes(a) + (b ? bytes(*b) : 0.0) <= (a.M <= 8 ? 28e6 : 16e6);
}

cudaError_t gemm_rows(const GemmArgs& a, const GemmArgs* b, const Dev& dev) {
  RowsDev p, q = {};
  if (!rows_dev(a, p) || (b && !rows_dev(*b, q))) return cudaErrorInvalidValue;
  const dim3 grid((unsigned)std::min(dev.num_sms, p.groups + q.groups)), block(kGrThreads);
  if (a.epi.act == ACT_SWIGLU)
    return a.M <= 8 ? launch_pdl(gemm_rows_kernel<1, true>, grid, block, 0, dev.stream, p, q)
                    : launch_pdl(gemm_rows_kernel<2, true>, grid, block, 0, dev.stream, p, q);
  return a.M <= 8 ? launch_pdl(gemm_rows_kernel<1, false>, grid, block, 0, dev.stream, p, q)
                  : launch_pdl(gemm_rows_kernel<2, false>, grid, block, 0, dev.stream, p, q);
}

}  // namespace adadsf
