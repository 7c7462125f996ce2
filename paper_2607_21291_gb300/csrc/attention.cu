// Eq. 1 among the kept tokens of each sequence, fp32 storage: softmax(Q K^T /
// sqrt(d_k)) V, causal in packed order. Kept positions ascend, so packed order
// is original order and "key j <= query i" is the original causal mask
// restricted to the kept set (Sec. 3.4: unselected tokens contribute no keys
// or values).
// (bf16 storage runs on the tensor cores: attention_tc.cu.)
//
// Past a few keys a block of 128 threads takes 64 queries of a head and walks the keys 64 at a
// time with an exact fp32 online softmax. Scores: thread (ty, tx) holds queries
// ty + 8 i and keys tx + 16 j (8 x 4), both operands read four features at a time
// from rows padded to spread over the banks; a warp owns 16 whole query rows, so
// row maxima and sums are shuffles and P passes through the warp's own part of
// shared memory. P V: the same 8 rows by 4 features (8 at a head width of 128). Twelve
// 16-byte shared loads feed 128 multiply-adds in either product, so shared memory
// bounds both at two thirds of the FMA rate. The next K tile loads during the
// softmax and P V, the next V tile during the scores. Blocks run longest rows
// first. One warp per query, which walked its keys one after another with a warp
// reduction each, took 186 us at 4 sequences of 383 tokens and 8 heads of 64;
// this takes 39 us (21 and 10 us at one sequence of 64 tokens).
#include <type_traits>

#include "common.cuh"
#include "internal.h"

namespace adadsf {
namespace {

constexpr int kAtQ = 64;         // queries of a block
constexpr int kAtK = 64;         // keys of a tile
constexpr int kAtThreads = 128;
constexpr int kAtPLd = kAtK + 4;

template <int HD>
struct AttnF32 {
  static constexpr int LD = HD + 4;                       // floats of a staged Q or K row
  static constexpr int FLOATS = (kAtQ + kAtK) * LD + kAtK * HD + kAtQ * kAtPLd;
  static constexpr int SMEM = FLOATS * 4;
};

template <int HD>
__global__ void __launch_bounds__(kAtThreads) attn_f32_kernel(const float* qkv, int64_t ldq, float* out, int64_t ldo,
                                                              int K, int n_heads, int n_kv, int B, float scale) {
  using C = AttnF32<HD>;
  constexpr int NO = HD / 64;   // 16-byte pieces of a thread's output columns
  extern __shared__ __align__(16) float smem_at[];
  float* sQ = smem_at;
  float* sK = sQ + kAtQ * C::LD;
  float* sV = sK + kAtK * C::LD;
  float* sP = sV + kAtK * HD;
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  const int nqb = (K + kAtQ - 1) / kAtQ;
  const int h = (int)(blockIdx.x % n_heads);
  const int b = (int)(blockIdx.x / n_heads % B);
  const int qb = nqb - 1 - (int)(blockIdx.x / n_heads / B);   // longest rows first
  const int q0 = qb * kAtQ;
  const int g = h / (n_heads / n_kv);
  const float* base = qkv + (int64_t)b * K * ldq;
  // 64 rows of HD floats from column c0 of packed rows r0 ...; rows past K become zeros
  auto load_rows = [&](float* dst, int ld, int64_t c0, int r0) {
#pragma unroll
    for (int i = 0; i < 64 * HD / 4 / kAtThreads; ++i) {
      const int v = i * kAtThreads + tid;
      const int r = v / (HD / 4), c = (v % (HD / 4)) * 4;
      const bool ok = r0 + r < K;
      cp_async16(smem_u32(dst + r * ld + c), base + (int64_t)(ok ? r0 + r : 0) * ldq + c0 + c, ok);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  const int64_t kc0 = (int64_t)n_heads * HD + (int64_t)g * HD, vc0 = kc0 + (int64_t)n_kv * HD;
  pdl_wait();
  load_rows(sQ, C::LD, (int64_t)h * HD, q0);
  load_rows(sK, C::LD, kc0, 0);
  load_rows(sV, HD, vc0, 0);
  float m[8], l[8];
  float4 o[8][NO];
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    m[i] = -INFINITY;
    l[i] = 0.f;
#pragma unroll
    for (int c = 0; c < NO; ++c) o[i][c] = make_float4(0.f, 0.f, 0.f, 0.f);
  }
  // O += P V for the tile's keys. DIAG: keys above a row's own are left out
  // altogether (their P is 0, but 0 times a later token's infinity is not).
  auto pv = [&](auto diag_c) {
    constexpr bool DIAG = decltype(diag_c)::value;
#pragma unroll 2
    for (int k = 0; k < kAtK; k += 4) {
      float4 pr[8];
#pragma unroll
      for (int i = 0; i < 8; ++i) pr[i] = *reinterpret_cast<const float4*>(sP + (ty + 8 * i) * kAtPLd + k);
#pragma unroll
      for (int e = 0; e < 4; ++e) {
#pragma unroll
        for (int c = 0; c < NO; ++c) {
          const float4 v = *reinterpret_cast<const float4*>(sV + (k + e) * HD + 64 * c + 4 * tx);
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            const float p = e == 0 ? pr[i].x : e == 1 ? pr[i].y : e == 2 ? pr[i].z : pr[i].w;
            if (!DIAG || k + e <= ty + 8 * i) {
              o[i][c].x = fmaf(p, v.x, o[i][c].x);
              o[i][c].y = fmaf(p, v.y, o[i][c].y);
              o[i][c].z = fmaf(p, v.z, o[i][c].z);
              o[i][c].w = fmaf(p, v.w, o[i][c].w);
            }
          }
        }
      }
    }
  };
  for (int j = 0; j <= qb; ++j) {
    asm volatile("cp.async.wait_group 1;" ::: "memory");   // K of this tile (and Q); V may be on its way
    __syncthreads();
    float s[8][4];
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
      for (int c = 0; c < 4; ++c) s[i][c] = 0.f;
#pragma unroll 2
    for (int k = 0; k < HD; k += 4) {
      float4 kv[4];
#pragma unroll
      for (int c = 0; c < 4; ++c) kv[c] = *reinterpret_cast<const float4*>(sK + (tx + 16 * c) * C::LD + k);
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const float4 q = *reinterpret_cast<const float4*>(sQ + (ty + 8 * i) * C::LD + k);
#pragma unroll
        for (int c = 0; c < 4; ++c)
          s[i][c] = fmaf(q.w, kv[c].w, fmaf(q.z, kv[c].z, fmaf(q.y, kv[c].y, fmaf(q.x, kv[c].x, s[i][c]))));
      }
    }
    __syncthreads();   // K is read: the next tile's may land
    if (j < qb) load_rows(sK, C::LD, kc0, (j + 1) * kAtK);
    else asm volatile("cp.async.commit_group;" ::: "memory");
    const bool diag = j == qb;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      float mx = -INFINITY;
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        s[i][c] *= scale;
        if (diag && tx + 16 * c > ty + 8 * i) s[i][c] = -INFINITY;
        mx = fmaxf(mx, s[i][c]);
      }
      const float m_new = fmaxf(m[i], max16(mx));
      const float a = expf(m[i] - m_new);
      float sum = 0.f;
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const float p = expf(s[i][c] - m_new);
        sum += p;
        sP[(ty + 8 * i) * kAtPLd + tx + 16 * c] = p;
      }
      l[i] = l[i] * a + sum16(sum);
      m[i] = m_new;
#pragma unroll
      for (int c = 0; c < NO; ++c) {
        o[i][c].x *= a;
        o[i][c].y *= a;
        o[i][c].z *= a;
        o[i][c].w *= a;
      }
    }
    asm volatile("cp.async.wait_group 1;" ::: "memory");   // V of this tile
    __syncthreads();                                        // V has landed for all; P is the warp's own
    if (diag) pdl_trigger();
    if (diag) pv(std::true_type());
    else pv(std::false_type());
    __syncthreads();   // V is read
    if (j < qb) load_rows(sV, HD, vc0, (j + 1) * kAtK);
  }
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int r = q0 + ty + 8 * i;
    if (r >= K) continue;
    float* dst = out + ((int64_t)b * K + r) * ldo + (int64_t)h * HD + 4 * tx;
#pragma unroll
    for (int c = 0; c < NO; ++c)
      *reinterpret_cast<float4*>(dst + 64 * c) =
          make_float4(o[i][c].x / l[i], o[i][c].y / l[i], o[i][c].z / l[i], o[i][c].w / l[i]);
  }
}

// Short sequences: a warp per (query, head, sequence), the lanes splitting the head,
// which walks its keys one after another. A tile of 64 queries and keys is mostly padding
// there, and this one's walk short: up to 8 keys, or 16 where the tiles are more than two
// an SM. us from a cold L2 / back to back, 8 heads of 64, tiles and this one:
//   1 sequence of 1 12.4 / 9.6, 8.3 / 4.3    of 8 13.4 / 10.4, 13.4 / 6.3    of 16 13.4 / 10.5, 19.6 / 8.4
//   64 sequences of 8 24.7 / 20.7, 14.5 / 8.3    of 16 24.7 / 20.8, 23.7 / 14.5    of 24 24.8 / 21.4, 37.0 / 20.4
//   512 sequences of 16 115 / 111, 85 / 52    of 24 117 / 113, 157 / 147
constexpr int kAtShort = 8, kAtShortMany = 16;

template <int HD>
__global__ void __launch_bounds__(kAtThreads)
    attn_f32_short_kernel(const float* qkv, int64_t ldq, float* out, int64_t ldo, int K, int n_heads, int n_kv,
                          int64_t n_warps, float scale) {
  pdl_wait();
  pdl_trigger();
  constexpr int PL = HD / 32;
  const int lane = threadIdx.x & 31;
  const int64_t wi = (int64_t)blockIdx.x * (kAtThreads / 32) + (threadIdx.x >> 5);
  if (wi >= n_warps) return;
  const int i = (int)(wi % K), h = (int)(wi / K % n_heads);
  const int64_t row0 = wi / K / n_heads * K;
  const int g = h / (n_heads / n_kv);
  const float* q = qkv + (row0 + i) * ldq + (int64_t)h * HD;
  const float* kr = qkv + row0 * ldq + (int64_t)(n_heads + g) * HD;
  const float* vr = kr + (int64_t)n_kv * HD;
  float qv[PL], o[PL];
#pragma unroll
  for (int e = 0; e < PL; ++e) {
    qv[e] = q[lane + 32 * e];
    o[e] = 0.f;
  }
  float m = -INFINITY, l = 0.f;
  for (int j = 0; j <= i; ++j, kr += ldq, vr += ldq) {
    float d = 0.f;
#pragma unroll
    for (int e = 0; e < PL; ++e) d = fmaf(qv[e], kr[lane + 32 * e], d);
    const float sc = warp_sum(d) * scale;
    const float m_new = fmaxf(m, sc);
    const float a = expf(m - m_new), p = expf(sc - m_new);
    l = l * a + p;
#pragma unroll
    for (int e = 0; e < PL; ++e) o[e] = o[e] * a + p * vr[lane + 32 * e];
    m = m_new;
  }
  float* dst = out + (row0 + i) * ldo + (int64_t)h * HD;
#pragma unroll
  for (int e = 0; e < PL; ++e) dst[lane + 32 * e] = o[e] / l;
}

template <int HD>
cudaError_t launch_attn_f32(const float* q, int64_t ld_qkv, float* o, int64_t ld_out, int B, int K, int n_heads,
                            int n_kv_heads, const Dev& dev) {
  const float scale = 1.f / sqrtf((float)HD);
  if (K <= kAtShort || (K <= kAtShortMany && (int64_t)B * n_heads > 2 * dev.num_sms)) {
    const int64_t warps = (int64_t)B * n_heads * K, nb = (warps + kAtThreads / 32 - 1) / (kAtThreads / 32);
    if (nb > INT32_MAX) return cudaErrorInvalidValue;
    return launch_pdl(attn_f32_short_kernel<HD>, dim3((unsigned)nb), dim3(kAtThreads), 0, dev.stream, q, ld_qkv, o, ld_out,
                      K, n_heads, n_kv_heads, warps, scale);
  }
  const int64_t blocks = (int64_t)((K + kAtQ - 1) / kAtQ) * n_heads * B;
  if (blocks > INT32_MAX) return cudaErrorInvalidValue;
  const cudaError_t e = allow_smem<attn_f32_kernel<HD>, AttnF32<HD>::SMEM>();
  if (e != cudaSuccess) return e;
  return launch_pdl(attn_f32_kernel<HD>, dim3((unsigned)blocks), dim3(kAtThreads), AttnF32<HD>::SMEM, dev.stream, q,
                    ld_qkv, o, ld_out, K, n_heads, n_kv_heads, B, scale);
}

}  // namespace

cudaError_t attention(int dtype, const void* qkv, int64_t ld_qkv, void* out, int64_t ld_out, int B,
                      int K, int n_heads, int n_kv_heads, int head_dim, const Dev& dev) {
  if (B <= 0 || K <= 0) return cudaSuccess;
  if (dtype != kF32) return cudaErrorInvalidValue;   // bf16 runs attention_tc
  const float* q = static_cast<const float*>(qkv);
  float* o = static_cast<float*>(out);
  if (head_dim == 64) return launch_attn_f32<64>(q, ld_qkv, o, ld_out, B, K, n_heads, n_kv_heads, dev);
  if (head_dim == 128) return launch_attn_f32<128>(q, ld_qkv, o, ld_out, B, K, n_heads, n_kv_heads, dev);
  return cudaErrorInvalidValue;
}

}  // namespace adadsf
