// Fused FP32 attention, forward and backward, in plain SIMT arithmetic: the paper's "fused FP32" comparison arm
// (Appendix "Accuracy and Cost", paragraph "Fused FP32 baseline"; Table "method-definitions", row "FP32 attention").
// It decodes the BF16 inputs, computes every product, the softmax and the gradients with FP32 fused multiply-adds on
// the CUDA cores (no tensor core, no TF32), returns BF16 outputs and gradients, and saves an FP32 output plus three
// FP32 row statistics (log-sum-exp, row maximum, inverse normaliser); nothing of size N^2 is stored.
//
//   fp32_attn_fwd_kernel   query tile stationary, online softmax over 64-key tiles (Eq. "row-attention")
//   fp32_attn_dq_kernel    query tile stationary:  D = rowsum(dO * O32), P = exp(s - max) / l, dS = P (dP - D), dQ = alpha dS K
//   fp32_attn_dkv_kernel   key tile stationary:    dV = P^T dO, dK = alpha dS^T Q            (Eq. "row-gradients")
//
// Layout.  A CTA owns 32 stationary rows and 8 warps.  A row lives in the registers of d / 32 neighbouring lanes, 32
// coordinates each (two rows per thread in the forward), together with its accumulators; the streamed rows lie in shared
// memory as FP32 and every lane of a warp reads the same row, so a dot product is 16 packed FMAs per lane and one or two
// shuffles, and neither P nor dS ever leaves the registers.  The warps that do not own other rows split the streamed rows
// between them (batches dealt round-robin) and their partial results are added up, in a fixed order, at the end: a tile of
// 32 rows keeps eight warps busy, and the longest causal tile is a 64th of a 2048-row head instead of a 32nd.
// What bounds it: a 16-byte shared-memory read with one or two distinct addresses takes 2 clk of the SM, four or more 4
// clk (microbenchmark), and feeds one packed FMA pair per row; with two rows per thread at d = 64 that is as much time as
// the FMAs.  Tiles wait in shared memory as BF16 (asynchronous copies) while the previous tile is in the ALUs.
// Measured, 4 heads x 2048 x 64, causal: forward 448 -> 84 us, backward 1644 -> 303 us; 3 heads x 1500 x 128: 709 -> 139
// and 2526 -> 614 us (before: 64-row tiles on four warps, 4 x 8 scores per thread with eight-way bank conflicts, P and dS
// through shared memory).
#pragma once
#include <cuda_bf16.h>
#include <stdint.h>

#include "sm100_primitives.cuh"

namespace gproj {

template <int D>
struct Fp32Cfg {
  static constexpr int kThreads = 256, kWarps = 8, kRows = 32, kTile = 64;
  static constexpr int kLanes = D / 32;                        // lanes per row
  static constexpr int kChunkF = 36, kRowF = kLanes * kChunkF; // a lane's 32 coordinates, padded by four banks
  static constexpr int kRawBytes = kTile * D * 2;              // one streamed tile as BF16
  static constexpr int kTileF = kTile * kRowF;                 // ... and as FP32
  static constexpr int kStatF = 4 * kTile;
  static constexpr int kMergeF = kRows * (D + 4);              // one partial accumulator of the tile
  static constexpr int kStreamSmem = 2 * kRawBytes + (2 * kTileF + kStatF) * 4;
  static constexpr int max_of(int a, int b) { return a > b ? a : b; }
  // warp grid: this many warps side by side over the 32 rows, the others over the streamed rows
  static constexpr int kFwdRpt = 2;                            // rows per thread in the forward (one in the backward)
  static constexpr int kFwdRowWarps = kRows / (32 / kLanes * kFwdRpt), kBwdRowWarps = kRows / (32 / kLanes);
  static constexpr int kFwdSmem = max_of(kStreamSmem, (kWarps / kFwdRowWarps) * (kMergeF + 2 * kRows) * 4);
  static constexpr int kDqSmem = max_of(kStreamSmem, (kWarps / kBwdRowWarps) * kMergeF * 4);
  static constexpr int kDkvSmem = max_of(kStreamSmem, (kWarps / kBwdRowWarps) * 2 * kMergeF * 4);
};

// Rows [row0, row0 + 64) of a [rows_total x D] BF16 matrix to shared memory, asynchronously; rows past the end as zeros.
// A thread later expands exactly the pieces it copied, so its own wait is enough.
template <int D>
__device__ __forceinline__ void fp32_fetch(uint8_t *raw, const __nv_bfloat16 *src, int row0, int rows_total) {
#pragma unroll
  for (int k = 0; k < 64 * (D / 8) / 256; ++k) {
    const int i = threadIdx.x + 256 * k, r = row0 + i / (D / 8), c8 = i % (D / 8);
    const __nv_bfloat16 *from = src + (r < rows_total ? static_cast<size_t>(r) * D + 8 * c8 : 0);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(smem_u32(raw + 16 * i)), "l"(from), "r"(r < rows_total ? 16 : 0) : "memory");
  }
}
__device__ __forceinline__ void fp32_fetch_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }
template <int D>
__device__ __forceinline__ void fp32_expand(float *tile, const uint8_t *raw) {
  using C = Fp32Cfg<D>;
#pragma unroll
  for (int k = 0; k < 64 * (D / 8) / 256; ++k) {
    const int i = threadIdx.x + 256 * k, r = i / (D / 8), c8 = i % (D / 8);
    const uint4 v = *reinterpret_cast<const uint4 *>(raw + 16 * i);
    float4 *o = reinterpret_cast<float4 *>(tile + r * C::kRowF + (c8 >> 2) * C::kChunkF + 8 * (c8 & 3));
    o[0] = make_float4(bf16_lo_to_f32(v.x), bf16_hi_to_f32(v.x), bf16_lo_to_f32(v.y), bf16_hi_to_f32(v.y));
    o[1] = make_float4(bf16_lo_to_f32(v.z), bf16_hi_to_f32(v.z), bf16_lo_to_f32(v.w), bf16_hi_to_f32(v.w));
  }
}
// 32 coordinates of one row from global memory as 16 packed pairs (zeros for a row that does not exist)
__device__ __forceinline__ void fp32_load_row(uint64_t (&x)[16], const __nv_bfloat16 *src, bool valid) {
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    const uint4 v = valid ? __ldg(reinterpret_cast<const uint4 *>(src) + c) : make_uint4(0u, 0u, 0u, 0u);
    const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int k = 0; k < 4; ++k) x[4 * c + k] = f32x2_bits(w[k] << 16, w[k] & 0xffff0000u);
  }
}
__device__ __forceinline__ float fp32_sum2(uint64_t v) {
  float a, b;
  f32x2_split(v, a, b);
  return a + b;
}
template <int D>
__device__ __forceinline__ float fp32_row_sum(float v) {      // over the lanes that share a row
#pragma unroll
  for (int o = 1; o < Fp32Cfg<D>::kLanes; o <<= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
// One partial accumulator row piece (32 coordinates) to the merge area
__device__ __forceinline__ void fp32_put(float *dst, const uint64_t (&x)[16], float scale) {
#pragma unroll
  for (int c = 0; c < 8; ++c) {
    float a, b, e, f;
    f32x2_split(x[2 * c], a, b);
    f32x2_split(x[2 * c + 1], e, f);
    reinterpret_cast<float4 *>(dst)[c] = make_float4(a * scale, b * scale, e * scale, f * scale);
  }
}
// BF16 rows from `parts` partial accumulators of the tile, added in order
template <int D>
__device__ __forceinline__ void fp32_merge_store(const float *parts, int n_parts, int part_stride, float scale, __nv_bfloat16 *dst, int row0, int rows_total) {
  for (int i = threadIdx.x; i < 32 * (D / 4); i += 256) {
    const int r = i / (D / 4), c4 = i % (D / 4);
    float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int g = 0; g < n_parts; ++g) {
      const float4 v = *reinterpret_cast<const float4 *>(parts + g * part_stride + r * (D + 4) + 4 * c4);
      s.x += v.x; s.y += v.y; s.z += v.z; s.w += v.w;
    }
    if (row0 + r < rows_total)
      *reinterpret_cast<uint2 *>(dst + static_cast<size_t>(row0 + r) * D + 4 * c4) = make_uint2(pack_bf16x2(s.x * scale, s.y * scale), pack_bf16x2(s.z * scale, s.w * scale));
  }
}

// saved state per (head, row): O32 [N][D], then lse, row maximum of the scaled scores, inverse normaliser ([N] each)
template <int D, bool CAUSAL>
__global__ void __launch_bounds__(256, 1) fp32_attn_fwd_kernel(const __nv_bfloat16 *__restrict__ Q, const __nv_bfloat16 *__restrict__ K,
                                                               const __nv_bfloat16 *__restrict__ V, __nv_bfloat16 *__restrict__ O,
                                                               float *__restrict__ O32, float *__restrict__ stats, int N, int BH, float alpha) {
  using C = Fp32Cfg<D>;
  constexpr int RPT = C::kFwdRpt, RG = C::kFwdRowWarps, SG = C::kWarps / RG, U = 4;
  extern __shared__ __align__(16) uint8_t fsm[];
  uint8_t *rawK = fsm, *rawV = rawK + C::kRawBytes;
  float *sK = reinterpret_cast<float *>(rawV + C::kRawBytes), *sV = sK + C::kTileF;
  // longest causal tiles first, all heads of a tile next to each other
  const int n_tiles = (N + 31) / 32, tile = n_tiles - 1 - static_cast<int>(blockIdx.x / BH), head = blockIdx.x % BH, q0 = 32 * tile;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, rg = warp % RG, sg = warp / RG, part = lane % C::kLanes;
  const int row_t = rg * (32 / RG) + (lane / C::kLanes) * RPT;                 // first of this thread's rows inside the tile
  const int warp_last = q0 + rg * (32 / RG) + 32 / RG - 1;
  const size_t hoff = static_cast<size_t>(head) * N * D;
  uint64_t q[RPT][16], o[RPT][16];
  float m_run[RPT], l_run[RPT];
#pragma unroll
  for (int i = 0; i < RPT; ++i) {
    fp32_load_row(q[i], Q + hoff + static_cast<size_t>(q0 + row_t + i) * D + 32 * part, q0 + row_t + i < N);
    m_run[i] = -INFINITY; l_run[i] = 0.f;
#pragma unroll
    for (int c = 0; c < 16; ++c) o[i][c] = 0ull;
  }
  const int kend = CAUSAL ? min(N, q0 + 32) : N;
  fp32_fetch<D>(rawK, K + hoff, 0, N);
  fp32_fetch<D>(rawV, V + hoff, 0, N);
  for (int k0 = 0; k0 < kend; k0 += 64) {
    fp32_fetch_wait();
    __syncthreads();                                           // the previous tile has been consumed
    fp32_expand<D>(sK, rawK);
    fp32_expand<D>(sV, rawV);
    __syncthreads();
    if (k0 + 64 < kend) {
      fp32_fetch<D>(rawK, K + hoff, k0 + 64, N);
      fp32_fetch<D>(rawV, V + hoff, k0 + 64, N);
    }
    const int last = min(kend, CAUSAL ? warp_last + 1 : N) - k0;                 // keys of the tile some row of the warp sees
    for (int b = U * sg; b < min(64, last); b += U * SG) {
      const float *kp = sK + b * C::kRowF + part * C::kChunkF, *vp = sV + b * C::kRowF + part * C::kChunkF;
      uint64_t s2[RPT][U];
#pragma unroll
      for (int i = 0; i < RPT; ++i)
#pragma unroll
        for (int u = 0; u < U; ++u) s2[i][u] = 0ull;
#pragma unroll
      for (int c = 0; c < 8; ++c)
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const ulonglong2 kk = *reinterpret_cast<const ulonglong2 *>(kp + u * C::kRowF + 4 * c);
#pragma unroll
          for (int i = 0; i < RPT; ++i) s2[i][u] = fma2(q[i][2 * c + 1], kk.y, fma2(q[i][2 * c], kk.x, s2[i][u]));
        }
      float p[RPT][U];
      bool raised = false;
      float m_new[RPT];
#pragma unroll
      for (int i = 0; i < RPT; ++i) {
        m_new[i] = m_run[i];
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const float s = fp32_row_sum<D>(fp32_sum2(s2[i][u])) * alpha;
          const int kj = k0 + b + u;
          p[i][u] = (kj < N && (!CAUSAL || kj <= q0 + row_t + i)) ? s : -INFINITY;
          m_new[i] = fmaxf(m_new[i], p[i][u]);
        }
        raised |= m_new[i] > m_run[i];
      }
      if (__any_sync(0xffffffffu, raised)) {
#pragma unroll
        for (int i = 0; i < RPT; ++i) {
          const float corr = (m_run[i] == -INFINITY) ? 0.f : __expf(m_run[i] - m_new[i]);
          const uint64_t c2 = f32x2(corr, corr);
          l_run[i] *= corr;
#pragma unroll
          for (int c = 0; c < 16; ++c) o[i][c] = mul2(o[i][c], c2);
          m_run[i] = m_new[i];
        }
      }
#pragma unroll
      for (int i = 0; i < RPT; ++i) {
        const float m = (m_run[i] == -INFINITY) ? 0.f : m_run[i];                // a row that has seen no key yet
#pragma unroll
        for (int u = 0; u < U; ++u) { p[i][u] = __expf(p[i][u] - m); l_run[i] += p[i][u]; }
      }
#pragma unroll
      for (int u = 0; u < U; ++u) {
        uint64_t p2[RPT];
#pragma unroll
        for (int i = 0; i < RPT; ++i) p2[i] = f32x2(p[i][u], p[i][u]);
#pragma unroll
        for (int c = 0; c < 8; ++c) {
          const ulonglong2 vv = *reinterpret_cast<const ulonglong2 *>(vp + u * C::kRowF + 4 * c);
#pragma unroll
          for (int i = 0; i < RPT; ++i) { o[i][2 * c] = fma2(p2[i], vv.x, o[i][2 * c]); o[i][2 * c + 1] = fma2(p2[i], vv.y, o[i][2 * c + 1]); }
        }
      }
    }
  }
  // merge of the SG partial softmaxes: O = sum_g o_g e_g / L, e_g = exp(m_g - M), L = sum_g l_g e_g
  __syncthreads();
  float *mm = reinterpret_cast<float *>(fsm), *ml = mm + SG * 32, *mo = ml + SG * 32;
  if (part == 0)
#pragma unroll
    for (int i = 0; i < RPT; ++i) { mm[sg * 32 + row_t + i] = m_run[i]; ml[sg * 32 + row_t + i] = l_run[i]; }
  __syncthreads();
#pragma unroll
  for (int i = 0; i < RPT; ++i) {
    float M = -INFINITY;
#pragma unroll
    for (int g = 0; g < SG; ++g) M = fmaxf(M, mm[g * 32 + row_t + i]);
    fp32_put(mo + sg * C::kMergeF + (row_t + i) * (D + 4) + 32 * part, o[i], (m_run[i] == -INFINITY) ? 0.f : __expf(m_run[i] - M));
  }
  __syncthreads();
  float *lse = stats + static_cast<size_t>(head) * 3 * N, *rmax = lse + N, *rinv = rmax + N;
  for (int i = threadIdx.x; i < 32 * (D / 4); i += 256) {
    const int r = i / (D / 4), c4 = i % (D / 4), qi = q0 + r;
    float M = -INFINITY, L = 0.f;
    for (int g = 0; g < SG; ++g) M = fmaxf(M, mm[g * 32 + r]);
    float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int g = 0; g < SG; ++g) {
      const float mg = mm[g * 32 + r];
      L += ml[g * 32 + r] * ((mg == -INFINITY) ? 0.f : __expf(mg - M));     // l is 0 without a key, and NaN where all scores were
      const float4 v = *reinterpret_cast<const float4 *>(mo + g * C::kMergeF + r * (D + 4) + 4 * c4);
      s.x += v.x; s.y += v.y; s.z += v.z; s.w += v.w;
    }
    const float inv = 1.f / L;
    s.x *= inv; s.y *= inv; s.z *= inv; s.w *= inv;
    if (qi < N) {
      *reinterpret_cast<float4 *>(O32 + hoff + static_cast<size_t>(qi) * D + 4 * c4) = s;
      *reinterpret_cast<uint2 *>(O + hoff + static_cast<size_t>(qi) * D + 4 * c4) = make_uint2(pack_bf16x2(s.x, s.y), pack_bf16x2(s.z, s.w));
      if (c4 == 0) { lse[qi] = M + __logf(L); rmax[qi] = M; rinv[qi] = inv; }
    }
  }
}

template <int D, bool CAUSAL>
__global__ void __launch_bounds__(256, 1) fp32_attn_dq_kernel(const __nv_bfloat16 *__restrict__ Q, const __nv_bfloat16 *__restrict__ K,
                                                              const __nv_bfloat16 *__restrict__ V, const __nv_bfloat16 *__restrict__ dO,
                                                              const float *__restrict__ O32, const float *__restrict__ stats,
                                                              float *__restrict__ Drow, __nv_bfloat16 *__restrict__ dQ, int N, int BH, float alpha) {
  using C = Fp32Cfg<D>;
  constexpr int RG = C::kBwdRowWarps, SG = C::kWarps / RG, U = 2;
  extern __shared__ __align__(16) uint8_t fsm[];
  uint8_t *rawK = fsm, *rawV = rawK + C::kRawBytes;
  float *sK = reinterpret_cast<float *>(rawV + C::kRawBytes), *sV = sK + C::kTileF;
  const int n_tiles = (N + 31) / 32, tile = n_tiles - 1 - static_cast<int>(blockIdx.x / BH), head = blockIdx.x % BH, q0 = 32 * tile;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, rg = warp % RG, sg = warp / RG, part = lane % C::kLanes;
  const int row_t = rg * (32 / RG) + lane / C::kLanes, qi = q0 + row_t, warp_last = q0 + rg * (32 / RG) + 32 / RG - 1;
  const size_t hoff = static_cast<size_t>(head) * N * D;
  const float *rmax = stats + static_cast<size_t>(head) * 3 * N + N, *rinv = rmax + N;
  const int kend = CAUSAL ? min(N, q0 + 32) : N;
  fp32_fetch<D>(rawK, K + hoff, 0, N);
  fp32_fetch<D>(rawV, V + hoff, 0, N);
  uint64_t q[16], u_[16], acc[16];
  fp32_load_row(q, Q + hoff + static_cast<size_t>(qi) * D + 32 * part, qi < N);
  fp32_load_row(u_, dO + hoff + static_cast<size_t>(qi) * D + 32 * part, qi < N);
  float dd = 0.f;                                              // D_i = sum_c dO_ic O_ic in FP32 from the FP32 output
  if (qi < N) {
    uint64_t d2 = 0ull;
    const ulonglong2 *o = reinterpret_cast<const ulonglong2 *>(O32 + hoff + static_cast<size_t>(qi) * D + 32 * part);
#pragma unroll
    for (int c = 0; c < 8; ++c) { const ulonglong2 v = o[c]; d2 = fma2(u_[2 * c + 1], v.y, fma2(u_[2 * c], v.x, d2)); }
    dd = fp32_sum2(d2);
  }
  dd = fp32_row_sum<D>(dd);
  if (sg == 0 && part == 0 && qi < N) Drow[static_cast<size_t>(head) * N + qi] = dd;
  const float mx = qi < N ? rmax[qi] : 0.f, inv = qi < N ? rinv[qi] : 0.f;
#pragma unroll
  for (int c = 0; c < 16; ++c) acc[c] = 0ull;
  for (int k0 = 0; k0 < kend; k0 += 64) {
    fp32_fetch_wait();
    __syncthreads();
    fp32_expand<D>(sK, rawK);
    fp32_expand<D>(sV, rawV);
    __syncthreads();
    if (k0 + 64 < kend) {
      fp32_fetch<D>(rawK, K + hoff, k0 + 64, N);
      fp32_fetch<D>(rawV, V + hoff, k0 + 64, N);
    }
    const int last = min(kend, CAUSAL ? warp_last + 1 : N) - k0;
    for (int b = U * sg; b < min(64, last); b += U * SG) {
      const float *kp = sK + b * C::kRowF + part * C::kChunkF, *vp = sV + b * C::kRowF + part * C::kChunkF;
      uint64_t kk[U][16], s2[U], p2[U], sb[U], pb[U];
#pragma unroll
      for (int u = 0; u < U; ++u) { s2[u] = p2[u] = sb[u] = pb[u] = 0ull; }
#pragma unroll
      for (int c = 0; c < 8; ++c)
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const ulonglong2 a = *reinterpret_cast<const ulonglong2 *>(kp + u * C::kRowF + 4 * c), v = *reinterpret_cast<const ulonglong2 *>(vp + u * C::kRowF + 4 * c);
          kk[u][2 * c] = a.x; kk[u][2 * c + 1] = a.y;
          s2[u] = fma2(q[2 * c], a.x, s2[u]); sb[u] = fma2(q[2 * c + 1], a.y, sb[u]);
          p2[u] = fma2(u_[2 * c], v.x, p2[u]); pb[u] = fma2(u_[2 * c + 1], v.y, pb[u]);
        }
      float ds[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const float s = fp32_row_sum<D>(fp32_sum2(add2(s2[u], sb[u]))), dp = fp32_row_sum<D>(fp32_sum2(add2(p2[u], pb[u])));
        const int kj = k0 + b + u;
        const bool keep = kj < N && (!CAUSAL || kj <= qi);
        ds[u] = keep ? __expf(fmaf(s, alpha, -mx)) * inv * (dp - dd) : 0.f;
      }
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const uint64_t d2 = f32x2(ds[u], ds[u]);
#pragma unroll
        for (int c = 0; c < 16; ++c) acc[c] = fma2(d2, kk[u][c], acc[c]);        // dQ += dS K
      }
    }
  }
  __syncthreads();
  float *mo = reinterpret_cast<float *>(fsm);
  fp32_put(mo + sg * C::kMergeF + row_t * (D + 4) + 32 * part, acc, 1.f);
  __syncthreads();
  fp32_merge_store<D>(mo, SG, C::kMergeF, alpha, dQ + hoff, q0, N);
}

template <int D, bool CAUSAL>
__global__ void __launch_bounds__(256, 1) fp32_attn_dkv_kernel(const __nv_bfloat16 *__restrict__ Q, const __nv_bfloat16 *__restrict__ K,
                                                               const __nv_bfloat16 *__restrict__ V, const __nv_bfloat16 *__restrict__ dO,
                                                               const float *__restrict__ stats, const float *__restrict__ Drow,
                                                               __nv_bfloat16 *__restrict__ dK, __nv_bfloat16 *__restrict__ dV, int N, int BH, float alpha) {
  using C = Fp32Cfg<D>;
  constexpr int RG = C::kBwdRowWarps, SG = C::kWarps / RG;
  extern __shared__ __align__(16) uint8_t fsm[];
  uint8_t *rawQ = fsm, *rawU = rawQ + C::kRawBytes;
  float *sQ = reinterpret_cast<float *>(rawU + C::kRawBytes), *sU = sQ + C::kTileF;
  float4 *sStat = reinterpret_cast<float4 *>(sU + C::kTileF);  // per streamed query: row maximum, inverse normaliser, D
  const int tile = static_cast<int>(blockIdx.x / BH), head = blockIdx.x % BH, k0 = 32 * tile;   // key tile 0 has the most queries (causal) and comes first
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, rg = warp % RG, sg = warp / RG, part = lane % C::kLanes;
  const int row_t = rg * (32 / RG) + lane / C::kLanes, kj = k0 + row_t;
  const size_t hoff = static_cast<size_t>(head) * N * D;
  const float *rmax = stats + static_cast<size_t>(head) * 3 * N + N, *rinv = rmax + N, *Dr = Drow + static_cast<size_t>(head) * N;
  const int q_first = CAUSAL ? k0 : 0;
  fp32_fetch<D>(rawQ, Q + hoff, q_first, N);
  fp32_fetch<D>(rawU, dO + hoff, q_first, N);
  uint64_t k[16], v[16], ak[16], av[16];
  fp32_load_row(k, K + hoff + static_cast<size_t>(kj) * D + 32 * part, kj < N);
  fp32_load_row(v, V + hoff + static_cast<size_t>(kj) * D + 32 * part, kj < N);
#pragma unroll
  for (int c = 0; c < 16; ++c) ak[c] = av[c] = 0ull;
  for (int q0 = q_first; q0 < N; q0 += 64) {
    float4 st = make_float4(0.f, 0.f, 0.f, 0.f);               // a query past the end has inverse normaliser 0: P = 0
    if (threadIdx.x < 64 && q0 + threadIdx.x < N) { const int qi = q0 + threadIdx.x; st = make_float4(rmax[qi], rinv[qi], Dr[qi], 0.f); }
    fp32_fetch_wait();
    __syncthreads();
    fp32_expand<D>(sQ, rawQ);
    fp32_expand<D>(sU, rawU);
    if (threadIdx.x < 64) sStat[threadIdx.x] = st;
    __syncthreads();
    if (q0 + 64 < N) {
      fp32_fetch<D>(rawQ, Q + hoff, q0 + 64, N);
      fp32_fetch<D>(rawU, dO + hoff, q0 + 64, N);
    }
    const int n = min(64, N - q0);
#pragma unroll 1
    for (int b = sg; b < n; b += SG) {
      const float *qp = sQ + b * C::kRowF + part * C::kChunkF, *up = sU + b * C::kRowF + part * C::kChunkF;
      const float4 t = sStat[b];
      uint64_t qq[16], uu[16], s2[2] = {0ull, 0ull}, p2[2] = {0ull, 0ull};
#pragma unroll
      for (int c = 0; c < 8; ++c) {
        const ulonglong2 a = *reinterpret_cast<const ulonglong2 *>(qp + 4 * c), e = *reinterpret_cast<const ulonglong2 *>(up + 4 * c);
        qq[2 * c] = a.x; qq[2 * c + 1] = a.y; uu[2 * c] = e.x; uu[2 * c + 1] = e.y;
        s2[0] = fma2(k[2 * c], a.x, s2[0]); s2[1] = fma2(k[2 * c + 1], a.y, s2[1]);
        p2[0] = fma2(v[2 * c], e.x, p2[0]); p2[1] = fma2(v[2 * c + 1], e.y, p2[1]);
      }
      const float s = fp32_row_sum<D>(fp32_sum2(add2(s2[0], s2[1]))), dp = fp32_row_sum<D>(fp32_sum2(add2(p2[0], p2[1])));
      const float p = (!CAUSAL || q0 + b >= kj) ? __expf(fmaf(s, alpha, -t.x)) * t.y : 0.f, ds = p * (dp - t.z);
      const uint64_t pp = f32x2(p, p), dd = f32x2(ds, ds);
#pragma unroll
      for (int c = 0; c < 16; ++c) { av[c] = fma2(pp, uu[c], av[c]); ak[c] = fma2(dd, qq[c], ak[c]); }   // dV += P^T dO, dK += dS^T Q
    }
  }
  __syncthreads();
  float *mo = reinterpret_cast<float *>(fsm);
  fp32_put(mo + (2 * sg) * C::kMergeF + row_t * (D + 4) + 32 * part, av, 1.f);
  fp32_put(mo + (2 * sg + 1) * C::kMergeF + row_t * (D + 4) + 32 * part, ak, 1.f);
  __syncthreads();
  fp32_merge_store<D>(mo, SG, 2 * C::kMergeF, 1.f, dV + hoff, k0, N);
  fp32_merge_store<D>(mo + C::kMergeF, SG, 2 * C::kMergeF, alpha, dK + hoff, k0, N);
}

}  // namespace gproj
