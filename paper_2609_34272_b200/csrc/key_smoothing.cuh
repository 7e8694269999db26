// Key smoothing, the comparison arm of Section 5.1 ("Key smoothing subtracts the per-document, per-KV-head mean key
// before calling the unmodified kernel ... autograd applies the matching correction to dK"), as one small HBM-bound
// kernel around the attention calls:
//
//   smooth_rows_kernel   Y_j = BF16(fl32(X_j - mean_j X_j))      X = K before the forward:  K~ = K - mean key
//                                                                X = dK~ after the backward: dK = dK~ - mean_j dK~_j,
//                        the vector-Jacobian product of the subtraction (in exact arithmetic sum_j dK~_j = 0,
//                        Proposition 3.1, so the second call removes only what rounding leaked into that sum).
//
// One CTA, or a cluster of 2, 4 or 8 (smooth_cluster in host_rules.h), per (head, sequence); all sequences of a call in one launch
// (the offsets travel as a kernel parameter).  A CTA reads its share of the rows twice, the second time from L2, with eight
// 16-byte loads per thread in flight, and the column sums of a cluster are exchanged through distributed shared memory.  Sums
// are FP32 in a fixed order, so results are reproducible.  Small calls are bound by the latency of one CTA (load, two
// exchanges, store), large ones by memory.  Keeping eight rows per thread in registers between the two passes instead needs
// 80 registers, with three CTAs on an SM instead of four, and loads the rows beyond them two at a time: measured, that -> this, in
// clusters of the same size, 64 x 32 heads x 1000 x 64: 149 -> 113 us; 4 x 32 x 4096 x 128: 122 -> 69; 24 documents, 19446 rows, 4 heads, d = 64:
// 12.8 -> 11.3; 8 heads x 300: the same.
#pragma once
#include <cuda_bf16.h>
#include <stdint.h>

#include "host_rules.h"
#include "sm100_primitives.cuh"

namespace gproj {

constexpr int kSmoothThreads = 256, kSmoothMaxSeqs = 512;   // at most kSmoothCtasPerSm CTAs run on an SM (host_rules.h)
struct SmoothOffsets { int cu[kSmoothMaxSeqs + 1]; };

// X, Y: [heads][rows_total][d] BF16; sequence blockIdx.x / (cluster size) of head blockIdx.y.
template <int D>
__global__ void __launch_bounds__(kSmoothThreads, kSmoothCtasPerSm)
smooth_rows_kernel(const __nv_bfloat16 *__restrict__ X, __nv_bfloat16 *__restrict__ Y, long long head_stride, const __grid_constant__ SmoothOffsets off) {
  constexpr int kLanes = D / 8;                       // threads across a row (8 BF16 = 16 bytes each)
  constexpr int kRowsPerPass = kSmoothThreads / kLanes, kWarps = kSmoothThreads / 32, kBatch = 8;
  __shared__ float part[kWarps][D];
  __shared__ __align__(16) float cta_sum[D];
  griddep_wait();
  griddep_launch_dependents();
  const int ncta = cluster_size(), rank = cluster_rank(), seq = blockIdx.x / ncta;
  const int row0 = off.cu[seq], rows = off.cu[seq + 1] - row0;
  const int per = (rows + ncta - 1) / ncta, r_begin = min(rows, rank * per), r_end = min(rows, r_begin + per);
  const int lane8 = threadIdx.x % kLanes, rsub = threadIdx.x / kLanes, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const long long base = static_cast<long long>(blockIdx.y) * head_stride + static_cast<long long>(row0) * D + 8 * lane8;
  const __nv_bfloat16 *x = X + base;
  __nv_bfloat16 *y = Y + base;
  float acc[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) acc[i] = 0.f;
  auto add = [&](const uint4 &v) {
    const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) { acc[2 * i] += bf16_lo_to_f32(w[i]); acc[2 * i + 1] += bf16_hi_to_f32(w[i]); }
  };
  uint4 batch[kBatch];
  auto fetch = [&](int r0) {
#pragma unroll
    for (int k = 0; k < kBatch; ++k) {
      const int r = r0 + k * kRowsPerPass;
      batch[k] = r < r_end ? *reinterpret_cast<const uint4 *>(x + static_cast<long long>(r) * D) : make_uint4(0u, 0u, 0u, 0u);
    }
  };
  for (int r = r_begin + rsub; r < r_end; r += kBatch * kRowsPerPass) {
    fetch(r);
#pragma unroll
    for (int k = 0; k < kBatch; ++k) add(batch[k]);
  }
  // column sums: over the rows of a warp, over the warps, over the cluster
#pragma unroll
  for (int o = kLanes; o < 32; o <<= 1)
#pragma unroll
    for (int i = 0; i < 8; ++i) acc[i] += __shfl_xor_sync(0xffffffffu, acc[i], o);
  if (lane < kLanes)
#pragma unroll
    for (int i = 0; i < 8; ++i) part[warp][8 * lane8 + i] = acc[i];
  __syncthreads();
  if (threadIdx.x < D) {
    float s = 0.f;
#pragma unroll
    for (int w = 0; w < kWarps; ++w) s += part[w][threadIdx.x];
    cta_sum[threadIdx.x] = s;
  }
  cluster_sync();
  float m[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) m[i] = 0.f;
#pragma unroll 4
  for (int c = 0; c < ncta; ++c) {
    const uint32_t remote = cluster_map_shared(smem_u32(&cta_sum[8 * lane8]), c);
    float v[8];
    cluster_load_f4(remote, v);
    cluster_load_f4(remote + 16, v + 4);
#pragma unroll
    for (int i = 0; i < 8; ++i) m[i] += v[i];
  }
#pragma unroll
  for (int i = 0; i < 8; ++i) m[i] /= static_cast<float>(rows);
  auto put = [&](int r, const uint4 &v) {
    const uint32_t w[4] = {v.x, v.y, v.z, v.w};
    uint32_t o[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) o[i] = pack_bf16x2(__fsub_rn(bf16_lo_to_f32(w[i]), m[2 * i]), __fsub_rn(bf16_hi_to_f32(w[i]), m[2 * i + 1]));
    *reinterpret_cast<uint4 *>(y + static_cast<long long>(r) * D) = make_uint4(o[0], o[1], o[2], o[3]);
  };
  for (int r0 = r_begin + rsub; r0 < r_end; r0 += kBatch * kRowsPerPass) {
    fetch(r0);
#pragma unroll
    for (int k = 0; k < kBatch; ++k) {
      const int r = r0 + k * kRowsPerPass;
      if (r < r_end) put(r, batch[k]);
    }
  }
  cluster_sync();                                     // no CTA leaves while another one may still read its sums
}

}  // namespace gproj
