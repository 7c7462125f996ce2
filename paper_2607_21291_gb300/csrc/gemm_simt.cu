// fp32 projections on CUDA cores (FFMA), for fp32 storage. TF32 tensor-core
// rounding would not hold the fp32 tolerance, so fp32 models take this path.
// Same epilogue semantics as the tensor-core kernel (see internal.h).
//
// Both operands are K-major. A stage holds 32 k of the tile's A and W rows as
// they lie in memory (16-byte asynchronous copies, three stages in flight,
// rows padded to 36 floats so that eight consecutive rows fall on different
// banks) and a thread reads four k of a row at once: TM + TN shared loads of
// 16 bytes feed 4 TM TN multiply-adds. A shared load of 16 bytes a lane takes
// four cycles, so shared memory bounds the narrow tile (8 x 4 a thread) at two
// thirds of the FMA rate; an 8 x 8 tile balances the two.
//
// What a projection of few rows lacks is CTAs and warps. Two splits along K give
// them: the KS thread groups of a block take 32 / KS of a stage's k each (their
// tiles are added in shared memory), and the S CTAs of a cluster take
// consecutive ranges of k, each finishing 1 / S of the tile's rows from the
// others' partial tiles in distributed shared memory. Both add in a fixed order.
//
// A GPT-NeoX layer's four projections are two launches, as on the tensor cores: QKV
// and MLP-up (one grid over both problems' tiles, the rotation in QKV's epilogue
// where a tile holds both halves of a pair), then output and MLP-down as two K
// sources of one sum. Against four launches, a rotary pass and a stored output
// projection: the Pythia-70M layer 69.0 -> 57.2 us on 128 tokens (64 kept), 350 ->
// 326 us on 4 x 511 (383 kept).
#include <math.h>

#include "common.cuh"
#include "internal.h"

namespace adadsf {
namespace {

struct SimtDev {
  const float* A; int64_t lda;
  const float* W; const float* W2; int64_t ldw;
  const float* A2; int64_t lda2;            // second K source: k >= K1 reads (A2, Wk2)
  const float* Wk2; int64_t ldwk2;
  int M, N, K, K1;                          // K: both sources together
  int act;
  const float* bias;
  const float* bias2;                       // added to bias, or null
  const float* add_packed; int64_t ld_add_packed;
  const float* add_rows; int64_t ld_add_rows;
  const int32_t* rows;
  int out_mapped;
  float* out; int64_t ld_out;
  const float* gate;                        // score gate (see internal.h), or null
  const float* gbase; int64_t ld_gbase;
  // rotary embedding of the first rope_cols columns (see internal.h; rope_half 0: off)
  const float2* rope_tab; const int32_t* rope_pos;
  int rope_T, rope_half, rope_hd, rope_cols;
};

constexpr int kF32Bk = 32;          // k of a stage
constexpr int kF32Ld = kF32Bk + 4;  // floats of a staged row
constexpr int kF32Stages = 3;

// BM x BN tile, TM x TN per thread, KS thread groups along k. DUAL: the first
// BN / 2 tile columns come from W, the others from W2 (same output columns).
template <int BM, int BN, int TM, int TN, int KS>
struct F32Tile {
  static constexpr int TX = BN / TN, TY = BM / TM;
  static constexpr int GROUP = TX * TY;
  static constexpr int THREADS = GROUP * KS;
  static constexpr int STAGE = (BM + BN) * kF32Ld;
  static constexpr int OLD = BN + 4;               // floats of a row of the finished tile
  static constexpr int RED = KS * BM * OLD;
  static constexpr int FLOATS = kF32Stages * STAGE > RED ? kF32Stages * STAGE : RED;
  static constexpr int SMEM = FLOATS * 4;
  static constexpr bool PACK = KS == 1;
  static_assert(TX == 8 && GROUP % 32 == 0, "lane layout");
  static_assert((BM + BN) * 8 % THREADS == 0 && THREADS % 8 == 0, "loader");
};

// Rotary partner of columns n .. n + 3: 0 if they do not rotate, else the distance to
// their pairs' other halves (the host fuses the rotation only where a half is whole
// groups of four columns and both halves lie in one tile).
__device__ __forceinline__ int rope_shift(const SimtDev& p, int n) {
  if (p.rope_half == 0 || n >= p.rope_cols) return 0;
  const int i = n % p.rope_hd;
  return i < p.rope_half ? p.rope_half : i < 2 * p.rope_half ? -p.rope_half : 0;
}

// Epilogue of columns n .. n + 3 of packed row m (acc: accumulator, acc2: the
// second weight's with DUAL, or the rotary partners' at columns n + shift).
template <bool DUAL>
__device__ __forceinline__ void f32_epilogue(const SimtDev& p, int m, int n, float4 acc, float4 acc2, int shift) {
  const int64_t arow = p.rows ? (int64_t)p.rows[m] : (int64_t)m;
  if (arow < 0) return;   // a row that bypasses the layer: nothing read or written
  const int64_t orow = p.out_mapped ? arow : (int64_t)m;
  float v[4] = {acc.x, acc.y, acc.z, acc.w};
  float f[4];
  if (p.bias) {
    load4(p.bias + n, f);
#pragma unroll
    for (int j = 0; j < 4; ++j) v[j] += f[j];
  }
  if (p.bias2) {
    load4(p.bias2 + n, f);
#pragma unroll
    for (int j = 0; j < 4; ++j) v[j] += f[j];
  }
  if (!DUAL && shift != 0) {
    float c[4] = {acc2.x, acc2.y, acc2.z, acc2.w};
    if (p.bias) {
      load4(p.bias + n + shift, f);
#pragma unroll
      for (int j = 0; j < 4; ++j) c[j] += f[j];
    }
    const int i = (shift > 0 ? n : n + shift) % p.rope_hd;
    const float2* cs = p.rope_tab + (int64_t)(p.rope_pos ? p.rope_pos[m] : m % p.rope_T) * p.rope_half + i;
    // first half: a cos - b sin; second half: b cos + a sin
#pragma unroll
    for (int j = 0; j < 4; ++j) v[j] = shift > 0 ? v[j] * cs[j].x - c[j] * cs[j].y : v[j] * cs[j].x + c[j] * cs[j].y;
  }
  if (DUAL) {
    const float u[4] = {acc2.x, acc2.y, acc2.z, acc2.w};
#pragma unroll
    for (int j = 0; j < 4; ++j) v[j] = v[j] / (1.f + expf(-v[j])) * u[j];
  } else if (p.act == ACT_GELU) {
#pragma unroll
    for (int j = 0; j < 4; ++j) v[j] = 0.5f * v[j] * (1.f + erff(v[j] * 0.70710678118654752f));
  }
  if (p.add_packed) {
    load4(p.add_packed + (int64_t)m * p.ld_add_packed + n, f);
#pragma unroll
    for (int j = 0; j < 4; ++j) v[j] += f[j];
  }
  if (p.gate) {
    const float g = 1.f / (1.f + expf(-p.gate[arow]));
    load4(p.gbase ? p.gbase + arow * p.ld_gbase + n : p.add_rows + arow * p.ld_add_rows + n, f);
#pragma unroll
    for (int j = 0; j < 4; ++j) v[j] = p.gbase ? fmaf(g, v[j] - f[j], f[j]) : fmaf(g, v[j], f[j]);
  } else if (p.add_rows) {
    load4(p.add_rows + arow * p.ld_add_rows + n, f);
#pragma unroll
    for (int j = 0; j < 4; ++j) v[j] += f[j];
  }
  *reinterpret_cast<float4*>(p.out + orow * p.ld_out + n) = make_float4(v[0], v[1], v[2], v[3]);
}

__device__ __forceinline__ void add4(float4& s, const float4& f) {
  s.x += f.x;
  s.y += f.y;
  s.z += f.z;
  s.w += f.w;
}

template <int BM, int BN, int TM, int TN, int KS, bool DUAL>
__global__ void __launch_bounds__(F32Tile<BM, BN, TM, TN, KS>::THREADS, 2)
    gemm_f32_kernel(const __grid_constant__ SimtDev pa, const __grid_constant__ SimtDev pb, int tiles_a, int S) {
  using C = F32Tile<BM, BN, TM, TN, KS>;
  constexpr int NOUT = DUAL ? BN / 2 : BN;         // output columns of a tile
  constexpr int LOADS = (BM + BN) * 8 / C::THREADS;
  constexpr int LROWS = C::THREADS / 8;            // rows a loading step covers
  extern __shared__ __align__(16) float smem_f32[];
  const int tid = threadIdx.x;
  // the first tiles_a tiles are problem a's, the rest b's
  const bool second_problem = (int)(blockIdx.x / S) >= tiles_a;
  const SimtDev& p = second_problem ? pb : pa;
  const int num_n = (p.N + NOUT - 1) / NOUT;
  const int tile = (int)(blockIdx.x / S) - (second_problem ? tiles_a : 0), rank = (int)(blockIdx.x % S);
  const int row0 = tile / num_n * BM, col0 = tile % num_n * NOUT;
  // this CTA's stages of 32 k
  const int nkb = (p.K + kF32Bk - 1) / kF32Bk;
  const int kb0 = (int)((int64_t)nkb * rank / S), kb1 = (int)((int64_t)nkb * (rank + 1) / S);
  // loader: 16-byte column lc of rows lr, lr + LROWS, ... of the stage (A rows, then W rows)
  const int lc = tid & 7, lr = tid >> 3;
  const uint32_t sbase = smem_u32(smem_f32);
  auto load_stage = [&](int kb, int slot) {
    const bool k2 = kb * kF32Bk >= p.K1;             // the second source (K1 is whole stages there)
    const int k = kb * kF32Bk + lc * 4 - (k2 ? p.K1 : 0);
    const bool kin = k < (k2 ? p.K - p.K1 : p.K1);
    const float* A = k2 ? p.A2 : p.A;
    const float* W = k2 ? p.Wk2 : p.W;
    const int64_t lda = k2 ? p.lda2 : p.lda, ldw = k2 ? p.ldwk2 : p.ldw;
    const uint32_t dst = sbase + 4u * (slot * C::STAGE + lr * kF32Ld + lc * 4);
#pragma unroll
    for (int i = 0; i < LOADS; ++i) {
      const int r = lr + i * LROWS;
      const float* src;
      bool ok;
      if (r < BM) {
        ok = row0 + r < p.M;
        src = A + (int64_t)(ok ? row0 + r : 0) * lda;
      } else {
        const int j = r - BM;
        const bool second = DUAL && j >= BN / 2;
        const int n = col0 + (second ? j - BN / 2 : j);
        ok = n < p.N;
        src = (second ? p.W2 : W) + (int64_t)(ok ? n : 0) * ldw;
      }
      ok = ok && kin;
      cp_async16(dst + 4u * (i * LROWS * kF32Ld), src + (kin ? k : 0), ok);
    }
  };
  pdl_wait();
#pragma unroll
  for (int s = 0; s < kF32Stages - 1; ++s) {
    if (kb0 + s < kb1) load_stage(kb0 + s, s);
    asm volatile("cp.async.commit_group;" ::: "memory");
  }
  const int grp = tid / C::GROUP, gt = tid % C::GROUP;
  const int tx = gt & 7, ty = gt >> 3;
  // PACK: the even and the odd k of a thread's sums in the two halves of a packed
  // multiply-add (half the issue slots, twice the accumulators)
  float2 acc[TM][TN];
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < TN; ++j) acc[i][j] = make_float2(0.f, 0.f);
  int slot = 0;
  for (int kb = kb0; kb < kb1; ++kb) {
    asm volatile("cp.async.wait_group %0;" ::"n"(kF32Stages - 2) : "memory");
    __syncthreads();   // the stage has landed for every thread; the slot refilled below is free
    {
      const int nxt = slot + kF32Stages - 1 >= kF32Stages ? slot - 1 : slot + kF32Stages - 1;
      if (kb + kF32Stages - 1 < kb1) load_stage(kb + kF32Stages - 1, nxt);
      asm volatile("cp.async.commit_group;" ::: "memory");
    }
    const float* As = smem_f32 + slot * C::STAGE + ty * kF32Ld + grp * (kF32Bk / KS);
    const float* Bs = smem_f32 + slot * C::STAGE + (BM + tx) * kF32Ld + grp * (kF32Bk / KS);
#pragma unroll
    for (int k = 0; k < kF32Bk / KS; k += 4) {
      float4 a[TM];
#pragma unroll
      for (int i = 0; i < TM; ++i) a[i] = *reinterpret_cast<const float4*>(As + i * C::TY * kF32Ld + k);
#pragma unroll
      for (int j = 0; j < TN; ++j) {
        const float4 b = *reinterpret_cast<const float4*>(Bs + j * C::TX * kF32Ld + k);
        if constexpr (C::PACK) {
#pragma unroll
          for (int i = 0; i < TM; ++i) acc[i][j] = __ffma2_rn(make_float2(a[i].x, a[i].y), make_float2(b.x, b.y), acc[i][j]);
#pragma unroll
          for (int i = 0; i < TM; ++i) acc[i][j] = __ffma2_rn(make_float2(a[i].z, a[i].w), make_float2(b.z, b.w), acc[i][j]);
        } else {
#pragma unroll
          for (int i = 0; i < TM; ++i) acc[i][j].x = fmaf(a[i].x, b.x, acc[i][j].x);
#pragma unroll
          for (int i = 0; i < TM; ++i) acc[i][j].x = fmaf(a[i].y, b.y, acc[i][j].x);
#pragma unroll
          for (int i = 0; i < TM; ++i) acc[i][j].x = fmaf(a[i].z, b.z, acc[i][j].x);
#pragma unroll
          for (int i = 0; i < TM; ++i) acc[i][j].x = fmaf(a[i].w, b.w, acc[i][j].x);
        }
      }
    }
    slot = slot + 1 == kF32Stages ? 0 : slot + 1;
  }
  asm volatile("cp.async.wait_all;" ::: "memory");
  pdl_trigger();
  __syncthreads();   // the finished tiles overlay the stages
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < TN; ++j)
      smem_f32[(grp * BM + ty + i * C::TY) * C::OLD + tx + j * C::TX] = C::PACK ? acc[i][j].x + acc[i][j].y : acc[i][j].x;
  __syncthreads();
  if (S > 1) {
    if (KS > 1) {
      // the groups' tiles into the first one
      for (int v = tid; v < BM * (BN / 4); v += C::THREADS) {
        float* q = smem_f32 + (v / (BN / 4)) * C::OLD + (v % (BN / 4)) * 4;
        float4 s = *reinterpret_cast<float4*>(q);
#pragma unroll
        for (int g = 1; g < KS; ++g) add4(s, *reinterpret_cast<float4*>(q + g * BM * C::OLD));
        *reinterpret_cast<float4*>(q) = s;
      }
    }
    cluster_sync();
  }
  const int rows_here = BM / S;   // rows [rank rows_here, ...) of the tile are finished here
  for (int v = tid; v < rows_here * (NOUT / 4); v += C::THREADS) {
    const int r = rank * rows_here + v / (NOUT / 4), c = (v % (NOUT / 4)) * 4;
    const int m = row0 + r, n = col0 + c;
    if (m >= p.M || n >= p.N) continue;
    float4 s = make_float4(0.f, 0.f, 0.f, 0.f), s2 = s;
    const int shift = DUAL ? BN / 2 : rope_shift(p, n);   // where the second operand's columns lie in the tile
    if (S == 1) {
#pragma unroll
      for (int g = 0; g < KS; ++g) {
        const float* q = smem_f32 + (g * BM + r) * C::OLD + c;
        add4(s, *reinterpret_cast<const float4*>(q));
        if (shift != 0) add4(s2, *reinterpret_cast<const float4*>(q + shift));
      }
    } else {
      const uint32_t q = sbase + 4u * (r * C::OLD + c);
      for (int w = 0; w < S; ++w) {
        const uint32_t qw = map_to_cta(q, w);
        add4(s, ld_cluster_f32x4(qw));
        if (shift != 0) add4(s2, ld_cluster_f32x4(qw + 4u * shift));
      }
    }
    f32_epilogue<DUAL>(p, m, n, s, s2, shift);
  }
  if (S > 1) cluster_sync();   // partial tiles stay until every CTA has read them
}

// Problem a, and b (M 0: none) of the same K in the same launch.
template <int BM, int BN, int TM, int TN, int KS, bool DUAL>
cudaError_t launch_f32(const SimtDev& a, const SimtDev& b, int S, const Dev& dev) {
  using C = F32Tile<BM, BN, TM, TN, KS>;
  constexpr int NOUT = DUAL ? BN / 2 : BN;
  auto tiles = [](const SimtDev& p) { return (((int64_t)p.M + BM - 1) / BM) * ((p.N + NOUT - 1) / NOUT); };
  const int64_t ctas = (tiles(a) + tiles(b)) * S;
  if (ctas > INT32_MAX) return cudaErrorInvalidValue;
  const cudaError_t e = allow_smem<gemm_f32_kernel<BM, BN, TM, TN, KS, DUAL>, C::SMEM>();
  if (e != cudaSuccess) return e;
  if (S == 1)
    return launch_pdl(gemm_f32_kernel<BM, BN, TM, TN, KS, DUAL>, dim3((unsigned)ctas), dim3(C::THREADS), C::SMEM,
                      dev.stream, a, b, (int)tiles(a), S);
  return launch_pdl_cluster(gemm_f32_kernel<BM, BN, TM, TN, KS, DUAL>, dim3((unsigned)ctas), dim3(C::THREADS), C::SMEM,
                            dev.stream, S, a, b, (int)tiles(a), S);
}

// Tile and split of a product: the fewest cycles over the CTAs that share an
// SM, two at a time (the large tile's four warps alone leave half of the SM's
// issue slots empty, and clusters land two CTAs on an SM as soon as they need
// more than half of the SMs). A CTA costs its multiply-adds at the tile's share of
// 128 a cycle (0.72 and 0.61, measured at M = 20000, N = K = 2048) and, per
// cluster size, what exchanging the partial tiles adds; the constants reproduce a
// sweep of both tiles and S = 1 ... 8 over 20 shapes to about 10 %. So few rows
// take the narrow tile split 4 or 8 ways (M = 64, N = 512, K = 2048: 38 us
// unsplit, 12 us at S = 4, 180 us before), and the large tile wins from about
// one CTA of it per SM (M = 1532, N = K / 4 = 512: 94 us narrow, 80 us large and
// split, 230 us before; M = 20000, N = K = 2048: 3.75 and 3.25 ms, 5.07 ms before).
struct F32Plan {
  bool large;
  int S;
};
template <bool DUAL>
F32Plan f32_plan(const SimtDev& a, const SimtDev& b, int num_sms) {
  const double exchange[4] = {0.0, 1500.0, 1600.0, 3000.0};   // cycles, S = 1, 2, 4, 8
  F32Plan best = {false, 1};
  double best_t = 1e300;
  const int nkb = (a.K + kF32Bk - 1) / kF32Bk;
  for (int t = 0; t < 2; ++t) {
    const int bm = t ? 128 : 64, bn = t ? 64 : 32;
    const int nout = DUAL ? bn / 2 : bn;
    auto count = [&](const SimtDev& p) { return (double)(((int64_t)p.M + bm - 1) / bm) * ((p.N + nout - 1) / nout); };
    const double tiles = count(a) + count(b);
    for (int i = 0, S = 1; i < 4 && S <= nkb; ++i, S *= 2) {
      const double work = (double)bm * bn * ((nkb + S - 1) / S * kF32Bk) / (128.0 * (t ? 0.72 : 0.61)) + exchange[i];
      const int share = t == 0 && (S == 1 || tiles * S <= 0.5 * num_sms) ? 1 : 2;   // CTAs an SM runs together
      const double x = tiles * S / (share * num_sms);
      const double cyc = share * work * (x <= 1.0 ? 1.0 : 0.5 * (x + ceil(x)));
      if (cyc < best_t) {
        best_t = cyc;
        best = {t == 1, S};
      }
    }
  }
  return best;
}

template <bool DUAL>
cudaError_t run_f32(const SimtDev& a, const SimtDev& b, const Dev& dev) {
  const F32Plan pl = f32_plan<DUAL>(a, b, dev.num_sms);
  return pl.large ? launch_f32<128, 64, 8, 8, 1, DUAL>(a, b, pl.S, dev) : launch_f32<64, 32, 8, 4, 4, DUAL>(a, b, pl.S, dev);
}

bool simt_dev(const GemmArgs& a, SimtDev& p) {
  if (a.a_gather || a.epi.nrm_psum) return false;
  if (a.K2 > 0 && (a.K % kF32Bk != 0 || a.W2)) return false;   // the sources meet on a stage
  p = SimtDev{};
  p.A = static_cast<const float*>(a.A); p.lda = a.lda;
  p.W = static_cast<const float*>(a.W); p.W2 = static_cast<const float*>(a.W2); p.ldw = a.ldw;
  p.A2 = static_cast<const float*>(a.A2); p.lda2 = a.lda2;
  p.Wk2 = static_cast<const float*>(a.Wk2); p.ldwk2 = a.ldwk2;
  p.M = (int)a.M; p.N = a.N; p.K = a.K + (a.K2 > 0 ? a.K2 : 0); p.K1 = a.K;
  p.act = a.epi.act;
  p.bias = static_cast<const float*>(a.epi.bias);
  p.bias2 = static_cast<const float*>(a.epi.bias2);
  if (p.bias2 && a.epi.rope_tab) return false;
  p.add_packed = static_cast<const float*>(a.epi.add_packed); p.ld_add_packed = a.epi.ld_add_packed;
  p.add_rows = static_cast<const float*>(a.epi.add_rows); p.ld_add_rows = a.epi.ld_add_rows;
  p.rows = a.epi.rows;
  p.out_mapped = a.epi.out_mapped ? 1 : 0;
  p.out = static_cast<float*>(a.epi.out); p.ld_out = a.epi.ld_out;
  p.gate = a.epi.gate_scores;
  p.gbase = static_cast<const float*>(a.epi.gate_base); p.ld_gbase = a.epi.ld_gate_base;
  if (a.epi.rope_tab) {
    if (!f32_fuses_rope(a.epi.rope_half, a.epi.rope_hd) || a.epi.act != ACT_NONE) return false;
    p.rope_tab = a.epi.rope_tab;
    p.rope_pos = a.epi.rope_pos;
    p.rope_T = a.epi.rope_T;
    p.rope_half = a.epi.rope_half;
    p.rope_hd = a.epi.rope_hd;
    p.rope_cols = a.epi.rope_cols;
  }
  return !(p.gate && (p.gbase ? p.add_rows != nullptr : p.add_rows == nullptr));
}

}  // namespace

// Both halves of every pair in one 32-column tile, in whole groups of four columns.
bool f32_fuses_rope(int half, int hd) { return half > 0 && half % 4 == 0 && 2 * half <= 32 && hd % 32 == 0; }

cudaError_t gemm_f32(const GemmArgs& a, const Dev& dev) {
  if (a.M <= 0) return cudaSuccess;
  SimtDev p, none = {};
  if (!simt_dev(a, p)) return cudaErrorInvalidValue;
  return a.epi.act == ACT_SWIGLU ? run_f32<true>(p, none, dev) : run_f32<false>(p, none, dev);
}

cudaError_t gemm_f32_grouped(const GemmArgs& a, const GemmArgs& b, const Dev& dev) {
  if (a.K != b.K || a.K2 > 0 || b.K2 > 0 || a.epi.act == ACT_SWIGLU || b.epi.act == ACT_SWIGLU) return cudaErrorInvalidValue;
  if (a.M <= 0) return gemm_f32(b, dev);
  if (b.M <= 0) return gemm_f32(a, dev);
  SimtDev p, q;
  if (!simt_dev(a, p) || !simt_dev(b, q)) return cudaErrorInvalidValue;
  return run_f32<false>(p, q, dev);
}

}  // namespace adadsf
