// Fused attention backward with the GProj correction for sm_100a (Algorithm 1).
//
// The work of Algorithm 1 is organised as two stationary kernels so that every accumulator lives
// in TMEM from its first to its last contribution (no atomics, no BF16 round trip, deterministic):
//
//   bwd_dq_kernel   query tile stationary; streams 64-key steps.  Per step: S = Q K^T, dP = dO V^T
//                   (tensor core -> TMEM), then per row (thread <-> TMEM lane): P = exp(S - LSE),
//                   r = BF16(P), t = BF16(P (dP - D)), rho += sum t, m += sum r (sums of the ROUNDED
//                   operands, Eq. "gproj-row-mass"), and two more contractions A += t K, B += r K with
//                   t, r read from TMEM.  Epilogue: lambda = rho / m (0 if m = 0),
//                   dQ = BF16(alpha (A - lambda B)) (Eq. "gproj-query-implemented"), and the scaled-query
//                   operand of the key correction, stored negated: Z = -BF16(lambda q).
//                   Also produces D = rowsum(dO * O) (Algorithm 1 line 1) and keeps it, with LSE in base
//                   two, for the second kernel.
//   bwd_dkv_kernel  key tile stationary; streams 64-query steps.  Per step: S^T = K Q^T, dP^T = V dO^T,
//                   r^T, t^T as above (thread <-> key row; LSE, D are per-column values from shared
//                   memory), dV += r^T dO, dK += t^T Q + r^T Z  -- the correction lands in the FP32
//                   accumulator before the final cast (Eq. "gproj-key-implemented").
//                   Epilogue: dK = BF16(alpha acc), dV = BF16(acc).
//
// Pipeline.  TMEM holds kNB score buffers (S and dP of one 64-wide step each) next to the two FP32
// accumulators: 3 buffers at d = 64, 2 at d = 128 (512 columns either way).  Four compute warpgroups form two
// groups; a group takes every second step and its two warpgroups split the step's 64 columns (thread <-> (row,
// 32-column slice)).  A buffer is back with the tensor core after half the ALU time one warpgroup per step would
// take -- that time bounds the loop  scores -> ALUs -> second-stage products -> buffer free  each buffer runs
// through -- while the two groups, at different phases, hide each other's TMEM and barrier latencies.
// The packed BF16 operands r / t overwrite the consumed S columns of their own 16-column chunk.
// The dK/dV kernel further splits a step's arithmetic in two phases with their own barriers (r^T from S^T first, then
// t^T from dP^T), so that dV += r^T dO and dK += r^T Z run on the tensor core while t^T is still being computed.  The tensor-core queue is only one or two instructions deep, so an issuing warp is stalled
// for as long as its MMAs execute and anything else it does (barrier polls, commits) would idle the pipe.
// Two warps therefore issue: warp 1 the score products of every step, warp 2 the second-stage products; each
// one's bookkeeping overlaps the other's MMAs.  Reuse of a score buffer is ordered by an explicit barrier
// (second-stage MMAs of step n committed -> scores of step n + kNB may be issued).
//
// Persistence.  One CTA per SM walks a static list of tiles: tiles are ordered by decreasing work and dealt
// to the CTAs in boustrophedon rounds, which balances causal work as well as a greedy scheduler would while
// staying deterministic and needing no counter.  Barrier set-up, the TMEM allocation and the launch latency
// are paid once; the step pipeline (stage ring, score buffers) runs on across tile boundaries, the stationary
// tile of the next work item is fetched by its own warp as soon as the last score product of the current one
// has been issued and completed, and a warpgroup of its own runs the epilogue of one tile during the first steps of the
// next.
#pragma once
#include "sm100_primitives.cuh"
#include "tile_schedule.h"

namespace gproj {

constexpr unsigned kFlagNoQCorrection = 1u;
constexpr unsigned kFlagNoKCorrection = 2u;

constexpr int kMaxSeqRows = 1 << 24;   // rows of a head (the entry points check it)

// Bytes of one 64-row block of the row-constant tile (64 rows x 16 BF16 columns).
constexpr int kExtBlockBytes = 2048;

template <int D>
struct BwdCfg {
  static constexpr int kSlabs = D / 64;
  static constexpr int kBigSlabBytes = 128 * 128;                 // 128-row slab (stationary tile)
  static constexpr int kBigTileBytes = kSlabs * kBigSlabBytes;
  static constexpr int kStepRows = 64;                            // rows of a streamed tile
  static constexpr int kStepSlabBytes = kStepRows * 128;
  static constexpr int kStepTileBytes = kSlabs * kStepSlabBytes;
  static constexpr int kNB = (D == 64) ? 3 : 2;                   // score buffers (steps in flight)
  // Compute warpgroups: kGroups groups of kSlices warpgroups.  Group a takes the steps g = a (mod kGroups); inside it
  // warpgroup h takes columns [kSliceCols h, kSliceCols (h + 1)) of the step.  Two groups keep two steps in the ALUs at
  // different phases (one group's TMEM / barrier latencies hide behind the other's arithmetic); two slices halve the
  // time a score buffer stays away from the tensor core.
  static constexpr int kGroups = 2, kSlices = 2;
  static constexpr int kWG = kGroups * kSlices;
  static constexpr int kSliceCols = kStepRows / kSlices;
  static constexpr int kCompute = 128 * kWG;                      // compute threads
  static constexpr int kThreads = 128 + kCompute;                 // stage producer, 2 MMA warps, tile loader; compute warpgroups
  // dQ-side kernel: one more warpgroup, which prepares the next tile's row constants and writes a finished tile out while
  // the compute warpgroups are already in the next one (before, 512 threads went through three barriers and the epilogue
  // together at each tile: 1.2-1.8 us at d = 64, 3.4 us at d = 128, with the tensor core idle but for the next tile's first
  // scores).  Measured, dQ side alone, before -> after: 16 packed documents of 16384 rows, 16 heads, d = 64: 169 -> 152 us;
  // 96 heads x 1000 x 128, causal: 88 -> 81 us; 16 heads x 4096 x 64, causal (3.5 tiles per CTA): 80.7 -> 79.0 us.
  // Registers: 768 x 80 at launch.  At d = 128 they are re-dealt 4 x 88 + 48 + 80 (80 for the compute warps spills there:
  // 4 heads x 16384: 519 us, with 88: 498 us); at d = 64 they stay as they are (re-dealt: 83 instead of 79 us, the step
  // loop is scheduled differently).
  static constexpr int kDqEpiWarp = 4 + 4 * kWG, kDqThreads = kThreads + 128;
  static constexpr bool kDqMoveRegs = (D == 128);
  static constexpr int kDqRegsCompute = 88, kDqRegsAux = 48, kDqRegsEpi = 80;
  static constexpr int kDkvEpiWarp = kDqEpiWarp, kDkvThreads = kDqThreads;   // the dK/dV side has the same extra warpgroup for its epilogue (80 registers)
  static_assert(kWG * kDqRegsCompute + kDqRegsAux + kDqRegsEpi <= 6 * 80, "register shares");
  // TMEM columns: buffer b holds S at 128 b and dP at 128 b + 64; accumulators follow
  static constexpr int kTmemCols = 512;
  static constexpr uint32_t kColAcc0 = 128 * kNB, kColAcc1 = 128 * kNB + D;
  static_assert(kColAcc1 + D <= 512, "TMEM budget");
  // dQ-side kernel: Q, dO resident; ring of (K, V) step tiles
  static constexpr int kDqStages = (D == 64) ? 6 : 4;
  static constexpr int kDqStageBytes = 2 * kStepTileBytes;
  static constexpr int kDqResBufs = (D == 64) ? 2 : 1;             // stationary (Q, dO) buffers
  static constexpr int kDqStagingBytes = 4 * 32 * 128;             // each epilogue warp: 32 rows x 64 columns of dQ
  static constexpr int kDqSmemBytes = kDqResBufs * 2 * kBigTileBytes + kDqStages * kDqStageBytes + kDqStagingBytes + 1024;
  // dK/dV-side kernel: K, V resident; ring of (Q, dO, Z, stats) step tiles
  static constexpr int kDkvStages = 3;                             // (this kernel runs at d = 128 only)
  static constexpr int kDkvStageBytes = 3 * kStepTileBytes + kExtBlockBytes;   // + the step's 64-row block of the row-constant tile
  static constexpr int kDkvStagingBytes = 4 * 32 * 64;             // each epilogue warp: 32 rows x 32 columns of dK or dV
  static constexpr int kDkvSmemBytes = 2 * kBigTileBytes + kDkvStages * kDkvStageBytes + kDkvStagingBytes + 1024;
  static_assert(kDqStages >= kNB + 1 && (D == 64 || kDkvStages >= kNB + 1), "a stage stays busy until its second-stage MMAs finish");
};

// Item number -> (rank of the tile in decreasing work, head).  Items are dealt in groups of `group` consecutive ranks of
// all heads; inside a group the ranks of one head are adjacent, so that CTAs running at the same time work on the same
// head and share the rows they stream (the other operand) in L2 instead of fetching one head each out of HBM.
// group = 1: every head's longest tile first (the exact longest-first order; packed calls, whose plan is already
// sorted); group = tiles per head: head-major (dense non-causal calls, whose tiles are all alike); in between for
// causal calls with many heads, where a few adjacent ranks differ little in work.
// Division of a non-negative 31-bit number by a divisor fixed at launch: quotient = umulhi(x, mul) >> shr (x itself if
// the divisor is 1), with L = ceil(log2 divisor), mul = ceil(2^(31 + L) / divisor) < 2^32 and shr = L - 1, set by the
// host.  Three instructions instead of the forty-odd of a division by a run-time value, which sat on every role's path
// at each tile.
struct FastDiv {
  unsigned div, mul, shr;
#ifdef __CUDACC__
  __device__ __forceinline__ int quot(int x) const {
    return div == 1u ? x : static_cast<int>(__umulhi(static_cast<unsigned>(x), mul) >> shr);
  }
#endif
};
struct ItemOrder {
  int gk, n_full;                   // ranks per group, full groups
  int solo;                         // CTAs with one item only (TileSched)
  FastDiv per_group, by_gk, by_rem; // items per group (heads x gk); ranks per group; ranks of the short last group
#ifdef __CUDACC__
  __device__ __forceinline__ void decode(int lin, int &rank, int &head) const {
    const int g = per_group.quot(lin), within = lin - g * static_cast<int>(per_group.div);
    const bool full = g < n_full;
    head = full ? by_gk.quot(within) : by_rem.quot(within);
    rank = g * gk + within - head * static_cast<int>(full ? by_gk.div : by_rem.div);
  }
  __device__ __forceinline__ int rank(int lin) const { int r, h; decode(lin, r, h); return r; }
  __device__ __forceinline__ int head(int lin) const { int r, h; decode(lin, r, h); return h; }
#endif
};

// One 128-row tile of one sequence.  Rows are counted inside a head ([heads][rows][d] tensors): dense calls have one
// sequence [0, N) per head; packed (variable-length) calls have several, listed tile by tile in a plan the host
// prepared, two int4 per tile: {row0, seq0, seq_end, blk0} with blk0 the first 64-row block of row statistics of the
// sequence's QUERIES, and {oseq0, oseq_end, -, -}.
// [oseq0, oseq_end) is the range of the OTHER operand's rows the tile works against (keys for a query tile, queries for a
// key tile); it differs from [seq0, seq_end) when query and key lengths are unequal.
struct TileInfo { int row0, seq0, seq_end, blk0, oseq0, oseq_end; };
__device__ __forceinline__ TileInfo tile_info(const int4 *plan, int idx, int dense_tile, int N, int N_other) {
  if (plan != nullptr) {
    const int4 e = __ldg(plan + 2 * idx), o = __ldg(plan + 2 * idx + 1);
    return TileInfo{e.x, e.y, e.z, e.w, o.x, o.y};
  }
  return TileInfo{128 * dense_tile, 0, N, 0, 0, N_other};
}
// Rows [row0, row0 + 128) may be written by a TMA store (which clips at the tensor's end N) unless the tile is the
// ragged tail of a sequence that is followed by another one.
__device__ __forceinline__ bool tile_store_by_tma(const TileInfo &t, int N) { return t.row0 + 128 <= t.seq_end || t.seq_end == N; }
// Plain row-wise copy of a staged [128 x D] BF16 tile (128-byte swizzled slabs) to global memory, rows < rows_valid only.
template <int D>
__device__ __forceinline__ void store_rows_clipped(const uint8_t *stage, int slab_bytes, __nv_bfloat16 *dst_row0, int row, int rows_valid) {
  if (row < rows_valid) {
    uint4 *dst = reinterpret_cast<uint4 *>(dst_row0 + static_cast<size_t>(row) * D);
#pragma unroll
    for (int ch = 0; ch < D / 8; ++ch)
      dst[ch] = *reinterpret_cast<const uint4 *>(stage + (ch >> 3) * slab_bytes + swz128_offset(row, ch & 7));
  }
}

enum BwdWaitCode {
  kDqWaitQ = 0x21, kDqWaitKV = 0x22, kDqWaitKVEmpty = 0x23, kDqWaitSdP = 0x24, kDqWaitTR = 0x25, kDqWaitAcc = 0x26, kDqWaitBuf = 0x27, kDqWaitResFree = 0x28, kDqWaitAccFree = 0x29, kDqWaitStats = 0x2a, kDqWaitMass = 0x2b, kDqWaitPeer = 0x2c,
  kDkvWaitKV = 0x31, kDkvWaitQ = 0x32, kDkvWaitQEmpty = 0x33, kDkvWaitSdP = 0x34, kDkvWaitTR = 0x35, kDkvWaitAcc = 0x36, kDkvWaitBuf = 0x37, kDkvWaitResFree = 0x38, kDkvWaitAccFree = 0x39, kDkvWaitPeer = 0x3a
};

// Arithmetic of one pair of adjacent score columns, shared by both kernels (Algorithm 1 lines 5-8):
//   p = exp2(x * (alpha log2 e) - LSE log2 e),  r = BF16(p),  t = BF16(fl32[p * fl32(dP - D)]).
// x2 / dp2 are the raw TMEM words of the two columns; nl2 = {-LSE log2 e} and nd2 = {-D} per column.
// keep0 / keep1 zero a probability beyond the causal diagonal.
template <bool MASKED>
__device__ __forceinline__ void score_pair(uint32_t x0, uint32_t x1, uint32_t dp0, uint32_t dp1, uint64_t scale2, uint64_t nl2,
                                           uint64_t nd2, bool keep0, bool keep1, uint32_t &r_packed, uint32_t &t_packed) {
  float a0, a1;
  f32x2_split(fma2(f32x2_bits(x0, x1), scale2, nl2), a0, a1);
  float p0 = fast_exp2(a0), p1 = fast_exp2(a1);
  if (MASKED) {
    if (!keep0) p0 = 0.f;
    if (!keep1) p1 = 0.f;
  }
  float t0, t1;
  f32x2_split(mul2(f32x2(p0, p1), add2(f32x2_bits(dp0, dp1), nd2)), t0, t1);
  r_packed = pack_bf16x2(p0, p1);
  t_packed = pack_bf16x2(t0, t1);
}

// One step of the dQ side for one query row and one slice (kSliceCols = 32 keys) of the step's 64 keys, in two 16-column
// chunks: the second chunk's TMEM load is in flight while the first is in the ALUs.  tS / tdP address the slice's S and
// dP columns; `lim` = (row index) - (key index of the slice's column 0): with MASKED, column c is beyond the causal
// diagonal (or past the last key) when c > lim.  The packed BF16 operands overwrite the chunk's OWN score columns (r over
// its first eight, t over its last eight: one K = 16 MMA slice each), so nobody writes over scores yet to be read.
template <bool MASKED>
__device__ __forceinline__ void dq_slice(uint32_t tS, uint32_t tdP, float scale_log2, float neg_lse2, float Dv, int lim,
                                         uint64_t &rho2, uint64_t &msum2) {
  const uint64_t scale2 = f32x2(scale_log2, scale_log2), nl2 = f32x2(neg_lse2, neg_lse2), nd2 = f32x2(-Dv, -Dv);
  uint32_t xs[2][16], xp[2][16];
  tmem_ld16(tS, xs[0]);
  tmem_ld16(tdP, xp[0]);
#pragma unroll
  for (int c = 0; c < 2; ++c) {
    tmem_wait_ld();
    if (c == 0) {
      tmem_ld16(tS + 16, xs[1]);
      tmem_ld16(tdP + 16, xp[1]);
    }
    uint32_t pr[8], pt[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int col = 16 * c + 2 * i;
      score_pair<MASKED>(xs[c][2 * i], xs[c][2 * i + 1], xp[c][2 * i], xp[c][2 * i + 1], scale2, nl2, nd2, col <= lim, col + 1 <= lim,
                         pr[i], pt[i]);
      // row masses of the operands AS ROUNDED (Eq. "gproj-row-mass"): re-expand the BF16 pairs and add in FP32
      msum2 = add2(msum2, f32x2_bits(pr[i] << 16, pr[i] & 0xffff0000u));
      rho2 = add2(rho2, f32x2_bits(pt[i] << 16, pt[i] & 0xffff0000u));
    }
    tmem_st8(tS + 16 * c, pr);
    tmem_st8(tS + 16 * c + 8, pt);
  }
}

// The dK/dV side does the arithmetic of a step in two phases, so that the tensor core can start on the products that need
// only r^T while the ALUs are still busy with t^T (measured: -15 % on that kernel at d = 128; the dQ side did not gain):
//   phase 1 (needs S^T):   p = exp2(x * (alpha log2 e) - LSE log2 e), r = BF16(p); p is kept in FP32 registers
//   phase 2 (needs dP^T):  t = BF16(fl32[p * fl32(dP - D)])
// Each thread owns one key row and one slice (32 query columns) of the step, handled in two 16-column chunks whose TMEM
// loads are software-pipelined; the packed operands overwrite the chunk's own consumed S columns (r the first eight, t
// the last eight).

// Phase 1 of the dK/dV side (thread <-> key row, columns = queries).  `lim` = (key row) - (query index of the slice's
// column 0): with MASKED, column c is a query before this key when c < lim; `hi` = (last query of the sequence) - (query
// index of column 0): a column c > hi belongs to the next packed sequence (or is zero fill).  The scores arrive as
// x - LSE / alpha: the score product carries one extra K = 16 slice (a constant matrix of ones times the step's
// row-constant tile), so no per-column constant has to be read here (every lane would need every column's value:
// broadcast reads from shared memory cost the 64-query kernel at d = 64 14 % when it still had them).
template <bool MASKED>
__device__ __forceinline__ void dkv_phase1(uint32_t tS, float scale_log2, int lim, int hi, float (&p)[32]) {
  const uint64_t scale2 = f32x2(scale_log2, scale_log2);
  uint32_t xs[2][16];
  tmem_ld16(tS, xs[0]);
#pragma unroll
  for (int c = 0; c < 2; ++c) {
    tmem_wait_ld();
    if (c == 0) tmem_ld16(tS + 16, xs[1]);
    uint32_t pr[8];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int col = 16 * c + 4 * i;
      float a[4];
      f32x2_split(mul2(f32x2_bits(xs[c][4 * i], xs[c][4 * i + 1]), scale2), a[0], a[1]);
      f32x2_split(mul2(f32x2_bits(xs[c][4 * i + 2], xs[c][4 * i + 3]), scale2), a[2], a[3]);
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        float pe = fast_exp2(a[e]);
        if (MASKED && (col + e < lim || col + e > hi)) pe = 0.f;
        p[col + e] = pe;
      }
      pr[2 * i] = pack_bf16x2(p[col], p[col + 1]);
      pr[2 * i + 1] = pack_bf16x2(p[col + 2], p[col + 3]);
    }
    tmem_st8(tS + 16 * c, pr);
  }
}

// Phase 2 of the dK/dV side.  The products arrive as dP - D (same extra slice as for the scores).
__device__ __forceinline__ void dkv_phase2(uint32_t tS, uint32_t tdP, const float (&p)[32]) {
  uint32_t xp[2][16];
  tmem_ld16(tdP, xp[0]);
#pragma unroll
  for (int c = 0; c < 2; ++c) {
    tmem_wait_ld();
    if (c == 0) tmem_ld16(tdP + 16, xp[1]);
    uint32_t pt[8];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int col = 16 * c + 4 * i;
      float t0, t1, t2, t3;
      f32x2_split(mul2(f32x2(p[col], p[col + 1]), f32x2_bits(xp[c][4 * i], xp[c][4 * i + 1])), t0, t1);
      f32x2_split(mul2(f32x2(p[col + 2], p[col + 3]), f32x2_bits(xp[c][4 * i + 2], xp[c][4 * i + 3])), t2, t3);
      pt[2 * i] = pack_bf16x2(t0, t1);
      pt[2 * i + 1] = pack_bf16x2(t2, t3);
    }
    tmem_st8(tS + 16 * c + 8, pt);
  }
}

// Row constants of one query row for the dK/dV side, which takes them through its score products instead of reading
// them per column.  Per 64-row block a K-major operand tile of 16 BF16 columns without swizzle (eight-row groups of 256
// bytes: the rows' first eight columns, then their last eight): columns 0..2 hold -LSE / alpha and columns 8..10 hold -D,
// each as three BF16 pieces whose sum is the FP32 value, the other columns zero.  A row with an empty support
// (LSE = +inf) gets a large finite value: its probabilities are zero either way, and an infinity would turn the zero
// entries of the constant operand into NaN.
__device__ __forceinline__ void write_row_constants(float *stats, size_t block, int row_in_block, float neg_lse2, float Dv, float scale_log2) {
  const float c = fmaxf(__fdiv_rn(neg_lse2, scale_log2), -1.0e30f), nd = -Dv;
  const uint32_t c0 = pack_bf16x2(c, 0.f), n0 = pack_bf16x2(nd, 0.f);
  const float c_r1 = c - bf16_lo_to_f32(c0), n_r1 = nd - bf16_lo_to_f32(n0);
  const uint32_t c1 = pack_bf16x2(c_r1, 0.f), n1 = pack_bf16x2(n_r1, 0.f);
  const uint32_t c2 = pack_bf16x2(c_r1 - bf16_lo_to_f32(c1), 0.f), n2 = pack_bf16x2(n_r1 - bf16_lo_to_f32(n1), 0.f);
  uint8_t *blk = reinterpret_cast<uint8_t *>(stats) + block * kExtBlockBytes + (row_in_block >> 3) * 256 + (row_in_block & 7) * 16;
  *reinterpret_cast<uint4 *>(blk) = make_uint4(c0 | (c1 << 16), c2, 0u, 0u);
  *reinterpret_cast<uint4 *>(blk + 128) = make_uint4(n0 | (n1 << 16), n2, 0u, 0u);
}

// D_i = sum_c dO_ic O_ic from the saved BF16 output, FP32 (Algorithm 1 line 1), of the ROWS tile rows from `r0` on, by one
// warp: 16-byte loads (D / 8 lanes share a row), eight elements by sequential FMAs, the partial sums by a butterfly.  Rows
// from `rows_valid` on get zero.
template <int D, int ROWS>
__device__ __forceinline__ void saved_output_dots(const __nv_bfloat16 *O, const __nv_bfloat16 *dO, int r0, int rows_valid, float *sD) {
  constexpr int L = D / 8, RPI = 32 / L, kIters = ROWS / RPI, kBatch = kIters < 4 ? kIters : 4;   // loads in flight per tensor
  const int lane = threadIdx.x & 31, sub = lane / L, part = lane % L;
#pragma unroll 1
  for (int it0 = 0; it0 < kIters; it0 += kBatch) {
    uint4 a[kBatch], b[kBatch];
#pragma unroll
    for (int it = 0; it < kBatch; ++it) {
      const int r = r0 + (it0 + it) * RPI + sub;
      a[it] = b[it] = make_uint4(0u, 0u, 0u, 0u);
      if (r < rows_valid) {
        a[it] = __ldg(reinterpret_cast<const uint4 *>(O + static_cast<size_t>(r) * D) + part);
        b[it] = __ldg(reinterpret_cast<const uint4 *>(dO + static_cast<size_t>(r) * D) + part);
      }
    }
#pragma unroll
    for (int it = 0; it < kBatch; ++it) {
      const uint32_t aw[4] = {a[it].x, a[it].y, a[it].z, a[it].w}, bw[4] = {b[it].x, b[it].y, b[it].z, b[it].w};
      float acc = 0.f;
#pragma unroll
      for (int w = 0; w < 4; ++w) {
        acc = fmaf(bf16_lo_to_f32(aw[w]), bf16_lo_to_f32(bw[w]), acc);
        acc = fmaf(bf16_hi_to_f32(aw[w]), bf16_hi_to_f32(bw[w]), acc);
      }
#pragma unroll
      for (int off = L / 2; off >= 1; off >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, off);
      if (part == 0) sD[r0 + (it0 + it) * RPI + sub] = acc;
    }
  }
}

// ============================================================================================
// dQ side
// ============================================================================================
// CL = 2: a cluster of two CTAs shares every tile: CTA r takes the key steps r, r + 2, ...; the row masses are exchanged, and CTA
// r gets both parts of A and B for its half of the columns (over the consumed Q / dO buffer), of which it writes dQ and Z.
// Used where whole tiles cannot be dealt evenly.
// SHORT: the compute warpgroups prepare the row constants of every tile, not of their first one only.  At d = 128 the extra
// warpgroup needs 4 us for those of one tile and 5 us for the epilogue of another, one after the other, and a tile of few steps is
// through the step loop sooner; the compute warps meanwhile wait for its Q and dO, which have a single buffer.  Measured, d = 128,
// off -> on (in brackets the kernel in which 512 threads did both): 64 x 16 heads x 128, causal: 80.3 -> 59.1 us (63.6); 64 x 16 x 500,
// causal: 371 -> 293 (302); 200 packed documents of 30 to 300 rows, 16 heads: 484 -> 302 (351); 8000 of 20 rows, 2 heads: 887 -> 628
// (535); but 16 x 16 x 700, not causal (11 steps a tile): 167 -> 182 (207).
template <int D, bool CAUSAL, int CL, bool SHORT>
__global__ void __launch_bounds__(BwdCfg<D>::kDqThreads, 1)
bwd_dq_kernel(const __grid_constant__ CUtensorMap tmQ,    // box 64 x 128 rows
              const __grid_constant__ CUtensorMap tmdO,   // box 64 x 128 rows
              const __grid_constant__ CUtensorMap tmK,    // box 64 x 64 rows
              const __grid_constant__ CUtensorMap tmV,    // box 64 x 64 rows
              const __nv_bfloat16 *__restrict__ Qg, const __nv_bfloat16 *__restrict__ Og, const __nv_bfloat16 *__restrict__ dOg,
              const float *__restrict__ LSE, float *__restrict__ stats,
              __nv_bfloat16 *__restrict__ dQg, __nv_bfloat16 *__restrict__ Zg,
              const int4 *__restrict__ plan, int nblk,                          // packed sequences: tile list; 64-row statistic blocks per head
              int N, int Nk, int BH, int Hq, int G, int total_tiles, const ItemOrder order, float scale_log2, float alpha, unsigned flags, int *status) {
  // N: query rows per head (own operand), Nk: key rows per head.  Causal support of query i: keys j <= i + (L_k - L_q).
  using C = BwdCfg<D>;
  constexpr int NB = C::kNB, R = C::kDqResBufs, S = C::kDqStages;
  constexpr long long kTileBudget = tile_wait_budget(kMaxSeqRows / C::kStepRows + 1);   // of a wait that may span a tile
  extern __shared__ uint8_t smem_raw[];
  uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t *sRes = smem;                                        // buffer rb: Q tile, then dO tile
  uint8_t *sKV = sRes + R * 2 * C::kBigTileBytes;              // stage s: K step tile, then V step tile
  uint8_t *sStaging = sKV + S * C::kDqStageBytes;              // epilogue warp w: 4096 w

  __shared__ uint64_t bar_res_full[R], bar_res_free[R], bar_kv_full[S], bar_kv_empty[S];
  __shared__ uint64_t bar_sdp_full[NB], bar_tr_ready[NB], bar_acc_done, bar_acc_free, bar_drain[2];
  __shared__ uint64_t bar_stats_ready[2], bar_mass_ready[2], bar_mass_free[2], bar_peer_mass, bar_peer_ready, bar_peer_full;
  __shared__ float s_peer[CL > 1 ? 4 : 1][128];          // the other CTA's rho and m, by tile parity
  __shared__ uint32_t tmem_base_smem;
  __shared__ int cta_abort, cta_skip;
  // per tile parity: row constants for the compute warpgroups, their row masses for the epilogue
  __shared__ float s_D[2][128], s_lse[2][128], s_rho[2][C::kWG][128], s_m[2][C::kWG][128];

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) cta_skip = *reinterpret_cast<volatile int *>(status);
  __syncthreads();
  if (CL == 1 && cta_skip != 0) { griddep_wait(); return; }   // an earlier wait gave up: drain the rest of the grid quickly (a cluster runs on with every wait falling through)

  // Ragged N: tiles and steps round up; rows past N load as zero (TMA fill) and are clipped on store.
  const int n_qt = (N + 127) / 128;
  AbortState ab{status, &cta_abort};
  if (threadIdx.x == 0) {
    cta_abort = CL > 1 ? cta_skip : 0;
    for (int r = 0; r < R; ++r) { mbar_init(&bar_res_full[r], 1); mbar_init(&bar_res_free[r], CL > 1 ? 1 + 128 : 1); }
    for (int p = 0; p < 2; ++p) { mbar_init(&bar_stats_ready[p], 128); mbar_init(&bar_mass_ready[p], C::kCompute); mbar_init(&bar_mass_free[p], 128); }
    for (int s = 0; s < S; ++s) { mbar_init(&bar_kv_full[s], 1); mbar_init(&bar_kv_empty[s], 1); }
    for (int b = 0; b < NB; ++b) { mbar_init(&bar_sdp_full[b], 1); mbar_init(&bar_tr_ready[b], 128 * C::kSlices); }
    mbar_init(&bar_acc_done, 1);
    mbar_init(&bar_peer_mass, 128); mbar_init(&bar_peer_ready, 1); mbar_init(&bar_peer_full, 128);
    mbar_init(&bar_acc_free, 128);
    mbar_init(&bar_drain[0], 1);
    mbar_init(&bar_drain[1], 1);
    fence_mbar_init();
  }
  if (warp == 1) { tmem_alloc(&tmem_base_smem, C::kTmemCols); tmem_relinquish(); }
  if (warp == 0 && lane == 0) {
    tma_prefetch_desc(&tmQ); tma_prefetch_desc(&tmdO); tma_prefetch_desc(&tmK); tma_prefetch_desc(&tmV);
  }
  tc_fence_before();
  if (CL > 1) cluster_sync(); else __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = __shfl_sync(0xffffffffu, tmem_base_smem, 0);   // the shuffle marks it warp-uniform

  // Everything so far may have run beside the kernel before this one in the stream; its memory is visible from here on.
  // The dK/dV-side kernel that follows may then be scheduled on SMs this kernel has left: its set-up and its
  // stationary-tile loads need nothing from here, and it waits (griddep_wait) before it reads the statistics and Z.
  griddep_wait();
  griddep_launch_dependents();

  TileSched sched(total_tiles, order.solo, CL);
  const int rank = CL > 1 ? cluster_rank() : 0;
  // tile decode: causal -> longest rows first
  auto tix = [&](int lin) { return order.rank(lin); };
  auto hix = [&](int lin) { return order.head(lin); };
  auto tile_of = [&](int lin) { return tile_info(plan, tix(lin), CAUSAL ? (n_qt - 1 - tix(lin)) : tix(lin), N, Nk); };
  // 64-key steps of a query tile: the keys its last row sees (causal) or all of them; at least one step, fully masked
  // if the tile sees no key at all, so that every tile runs through the same pipeline.
  auto steps_of = [&](const TileInfo &t) {
    const int Lk = t.oseq_end - t.oseq0, off = Lk - (t.seq_end - t.seq0);
    const int kend = CAUSAL ? min(Lk, t.row0 - t.seq0 + 128 + off) : Lk;
    return max(1, (max(kend, 0) + C::kStepRows - 1) / C::kStepRows);
  };
  // This CTA's steps of a tile with T steps, and the n-th of them; a CTA that gets none runs step 0 fully masked.
  auto own_steps = [&](int T) { return CL == 1 ? T : max(1, (T - rank + CL - 1) / CL); };
  auto own_step = [&](int n, int T) { return CL == 1 ? n : (rank < T ? CL * n + rank : 0); };

  if (warp < 4) {
  if constexpr (C::kDqMoveRegs) setmaxnreg_dec<C::kDqRegsAux>();
  if (warp == 0) {
    // ---------------------------------------------------------------- TMA producer of the streamed (K, V) step tiles
    if (lane == 0) {
      int g = 0;
      for (int lin = sched.next(); lin >= 0; lin = sched.next()) {
        const TileInfo tl = tile_of(lin);
        const int bh = hix(lin), T = steps_of(tl);
        for (int m = 0; m < own_steps(T); ++m, ++g) {
          const int st = g % S, n = own_step(m, T);
          if (g >= S) mbar_wait(&bar_kv_empty[st], ((g / S) - 1) & 1, ab, kDqWaitKVEmpty);
          mbar_expect_tx(&bar_kv_full[st], C::kDqStageBytes);
          uint8_t *dst = sKV + st * C::kDqStageBytes;
          const int kvh = kv_head_of(bh, Hq, G), krow = tl.oseq0 + n * C::kStepRows;   // grouped-query: the group's shared K / V head
          for (int s = 0; s < C::kSlabs; ++s) {
            tma_load_3d(dst + s * C::kStepSlabBytes, &tmK, &bar_kv_full[st], s * 64, krow, kvh);
            tma_load_3d(dst + C::kStepTileBytes + s * C::kStepSlabBytes, &tmV, &bar_kv_full[st], s * 64, krow, kvh);
          }
        }
      }
      // Every load is consumed by an MMA the epilogue waits for, so nothing is in flight at exit unless the
      // CTA aborted; then give the copies a bounded chance to land before shared memory is released.
      if (cta_abort) {
        for (int q = (g > S ? g - S : 0); q < g; ++q)
          for (int spin = 0; spin < 100000 && !mbar_try_wait(&bar_kv_full[q % S], (q / S) & 1); ++spin) {}
      }
    }
  } else if (warp == 3) {
    // ---------------------------------------------------------------- TMA loader of the stationary (Q, dO) tiles
    if (lane == 0) {
      int ti = 0;
      for (int lin = sched.next(); lin >= 0; lin = sched.next(), ++ti) {
        const int rb = ti % R, bh = hix(lin);
        const TileInfo tl = tile_of(lin);
        if (ti >= R) mbar_wait(&bar_res_free[rb], ((ti / R) - 1) & 1, ab, kDqWaitResFree, kTileBudget);
        mbar_expect_tx(&bar_res_full[rb], 2 * C::kBigTileBytes);
        uint8_t *dst = sRes + rb * 2 * C::kBigTileBytes;
        for (int s = 0; s < C::kSlabs; ++s) {
          tma_load_3d(dst + s * C::kBigSlabBytes, &tmQ, &bar_res_full[rb], s * 64, tl.row0, bh);
          tma_load_3d(dst + C::kBigTileBytes + s * C::kBigSlabBytes, &tmdO, &bar_res_full[rb], s * 64, tl.row0, bh);
        }
      }
      if (cta_abort)
        for (int q = (ti > R ? ti - R : 0); q < ti; ++q)
          for (int spin = 0; spin < 100000 && !mbar_try_wait(&bar_res_full[q % R], (q / R) & 1); ++spin) {}
    }
  } else if (warp == 1) {
    // ---------------------------------------------------------------- tensor-core issuer 1: scores
    // The whole warp runs this loop so that every address stays provably warp-uniform (descriptor operands
    // then live in uniform registers); one elected lane issues the MMAs and commits.
    constexpr uint32_t idesc_s = idesc_bf16_f32(128, 64, 0, 0);    // [128 queries] x [64 keys], contraction over d
    const SmemDesc dscRes0 = make_smem_desc(smem_u32(sRes), 16, 1024);
    const SmemDesc dscK0 = make_smem_desc(smem_u32(sKV), 16, 1024);                          // K-major view of stage 0
    int g = 0, ti = 0;
    for (int lin = sched.next(); lin >= 0; lin = sched.next(), ++ti) {
      const int T = own_steps(steps_of(tile_of(lin))), rb = ti % R;
      mbar_wait(&bar_res_full[rb], (ti / R) & 1, ab, kDqWaitQ);
      const SmemDesc dscQ = dscRes0.advanced(rb * 2 * C::kBigTileBytes), dscdO = dscQ.advanced(C::kBigTileBytes);
      for (int n = 0; n < T; ++n, ++g) {
        const int st = g % S, b = g % NB;
        mbar_wait(&bar_kv_full[st], (g / S) & 1, ab, kDqWaitKV);
        // r, t of step g - NB consumed: that step's second-stage products are complete.  One commit per step serves this
        // wait and the stage ring's (every commit costs the tensor pipe some forty cycles in this stream of short products).
        if (g >= NB) mbar_wait(&bar_kv_empty[(g - NB) % S], ((g - NB) / S) & 1, ab, kDqWaitBuf);
        tc_fence_after();
        const SmemDesc dscK = dscK0.advanced(st * C::kDqStageBytes), dscV = dscK.advanced(C::kStepTileBytes);
        const uint32_t tS = tmem_base + 128 * b, tdP = tS + 64;
        if (elect_one_sync()) {
#pragma unroll
          for (int k = 0; k < D / 16; ++k) {
            const uint32_t oa = (k / 4) * C::kBigSlabBytes + (k % 4) * 32, ob = (k / 4) * C::kStepSlabBytes + (k % 4) * 32;
            umma_ss(tS, dscQ.at(oa), dscK.at(ob), idesc_s, k > 0);
          }
#pragma unroll
          for (int k = 0; k < D / 16; ++k) {
            const uint32_t oa = (k / 4) * C::kBigSlabBytes + (k % 4) * 32, ob = (k / 4) * C::kStepSlabBytes + (k % 4) * 32;
            umma_ss(tdP, dscdO.at(oa), dscV.at(ob), idesc_s, k > 0);
          }
          umma_commit(&bar_sdp_full[b]);
          if (n == T - 1) umma_commit(&bar_res_free[rb]);   // no MMA reads this Q / dO buffer any more
        }
        __syncwarp();
      }
    }
    drain_mmas_if_aborted(&bar_drain[0], ab);
  } else if (warp == 2) {
    // ---------------------------------------------------------------- tensor-core issuer 2: A += t K, B += r K
    constexpr uint32_t idesc_a = idesc_bf16_f32(128, D, 0, 1);     // [128 queries] x [d], contraction over 64 keys
    const SmemDesc dscK0mn = make_smem_desc(smem_u32(sKV), C::kStepSlabBytes, 1024);       // MN-major view of stage 0
    int g = 0, ti = 0;
    for (int lin = sched.next(); lin >= 0; lin = sched.next(), ++ti) {
      const int T = own_steps(steps_of(tile_of(lin)));
      if (ti > 0) mbar_wait(&bar_acc_free, (ti - 1) & 1, ab, kDqWaitAccFree);   // the previous epilogue has read A, B
      for (int p = 0; p < T; ++p, ++g) {
        const int st = g % S, b = g % NB;
        mbar_wait(&bar_tr_ready[b], (g / NB) & 1, ab, kDqWaitTR);
        tc_fence_after();
        const SmemDesc dscK = dscK0mn.advanced(st * C::kDqStageBytes);
        // packed BF16 operands of key slice k (16 keys): r over columns 16 k .. 16 k + 7 of the buffer, t over the next eight
        const uint32_t tR = tmem_base + 128 * b, tT = tR + 8;
        const uint32_t acc = (p > 0) ? 1u : 0u;
        if (elect_one_sync()) {
#pragma unroll
          for (int k = 0; k < C::kStepRows / 16; ++k)
            umma_ts(tmem_base + C::kColAcc0, tT + 16 * k, dscK.at(k * 2048), idesc_a, k > 0 ? 1u : acc);
#pragma unroll
          for (int k = 0; k < C::kStepRows / 16; ++k)
            umma_ts(tmem_base + C::kColAcc1, tR + 16 * k, dscK.at(k * 2048), idesc_a, k > 0 ? 1u : acc);
          umma_commit(&bar_kv_empty[st]);                   // step done: its stage and its score buffer are free
          if (p == T - 1) umma_commit(&bar_acc_done);
        }
        __syncwarp();
      }
    }
    drain_mmas_if_aborted(&bar_drain[1], ab);
  }
  } else if (warp < C::kDqEpiWarp) {
    // ---------------------------------------------------------------- compute: thread <-> (query row, key slice of every kGroups-th step)
    if constexpr (C::kDqMoveRegs) setmaxnreg_inc<C::kDqRegsCompute>();
    const int wg = (warp - 4) >> 2, grp = wg / C::kSlices, slice = wg % C::kSlices;
    const int row = 32 * (warp & 3) + lane;
    const uint32_t lane_addr = static_cast<uint32_t>(32 * (warp & 3)) << 16;
    const uint32_t slice_addr = tmem_base + lane_addr + C::kSliceCols * slice;
    int g0 = 0, ti = 0;
    for (int lin = sched.next(); lin >= 0; lin = sched.next(), ++ti) {
      const TileInfo tl = tile_of(lin);
      const int Tall = steps_of(tl), T = own_steps(Tall), par = ti & 1;
      const int qrow = tl.row0 + row;                  // this thread's query row within the head (past seq_end in a ragged tile)
#ifdef GPROJ_TRACE
      const unsigned long long ev_n0 = global_ns(); const long long ev_c0 = clock64(); unsigned long long ev_n1 = 0, ev_n2 = 0;
#endif
      if (SHORT || ti == 0) {
        // The first tile's constants come from these warps, which have nothing else to do yet, and so do a short one's.  They
        // overwrite those of tile ti - 2, whose readers have all handed in their row masses.
        if (SHORT && ti >= 2) mbar_wait(&bar_mass_ready[par], ((ti >> 1) - 1) & 1, ab, kDqWaitMass, kTileBudget);
        constexpr int kRows = 128 / (4 * C::kWG);
        const int cp = SHORT ? par : 0;
        const size_t row0 = static_cast<size_t>(hix(lin)) * N + tl.row0;
        const float lse_row = (qrow < tl.seq_end) ? LSE[row0 + row] : 0.f;
        saved_output_dots<D, kRows>(Og + row0 * D, dOg + row0 * D, kRows * (warp - 4), tl.seq_end - tl.row0, s_D[cp]);
        named_bar_sync(1, C::kCompute);
        if (wg == 0) {
          s_lse[cp][row] = lse_row;
          const int rel = qrow - tl.seq0;
          if (rank == 0 && rel < ((tl.seq_end - tl.seq0 + 63) / 64) * 64)
            write_row_constants(stats, static_cast<size_t>(hix(lin)) * nblk + tl.blk0 + (rel >> 6), rel & 63, -lse_row * 1.4426950408889634f, s_D[cp][row], scale_log2);
          mbar_arrive(&bar_stats_ready[cp]);
        }
      }
      mbar_wait(&bar_stats_ready[par], (ti >> 1) & 1, ab, kDqWaitStats);
      const float Dv = s_D[par][row], neg_lse2 = -s_lse[par][row] * 1.4426950408889634f;

      uint64_t rho2 = f32x2(0.f, 0.f), msum2 = f32x2(0.f, 0.f);
#ifdef GPROJ_TRACE
      ev_n1 = global_ns();
#endif
      for (int n = (grp - g0 % C::kGroups + C::kGroups) % C::kGroups; n < T; n += C::kGroups) {
        const int g = g0 + n, b = g % NB;
        mbar_wait(&bar_sdp_full[b], (g / NB) & 1, ab, kDqWaitSdP);
        tc_fence_after();
        const uint32_t tS16 = slice_addr + 128 * b, tdP16 = tS16 + 64;
        // Probabilities are zeroed beyond the causal diagonal and, in the ragged last step, for the zero-filled keys
        // past N (which would otherwise enter the row masses).  Rows of a causal tile never reach such keys.
        const int Lk = tl.oseq_end - tl.oseq0, off = Lk - (tl.seq_end - tl.seq0);
        const int ns = own_step(n, Tall);
        const bool none = CL > 1 && rank >= Tall;                            // a step of the other CTA, run to keep the pipeline in step
        const int krel0 = ns * C::kStepRows + C::kSliceCols * slice;         // key (inside its sequence) of the slice's column 0
        const bool masked = (CAUSAL && (ns + 1) * C::kStepRows - 1 > tl.row0 - tl.seq0 + off) || (ns + 1) * C::kStepRows > Lk || none;
        if (masked) {
          const int lim_c = CAUSAL ? qrow - tl.seq0 + off - krel0 : (1 << 30);
          dq_slice<true>(tS16, tdP16, scale_log2, neg_lse2, Dv, none ? -1 : min(lim_c, Lk - 1 - krel0), rho2, msum2);
        } else {
          dq_slice<false>(tS16, tdP16, scale_log2, neg_lse2, Dv, 0, rho2, msum2);
        }
        tmem_wait_st();
        tc_fence_before();
        mbar_arrive(&bar_tr_ready[b]);
      }
#ifdef GPROJ_TRACE
      ev_n2 = global_ns();
#endif
      // hand this warpgroup's share of the row masses to the epilogue and go on with the next tile
      float rho_lo, rho_hi, m_lo, m_hi;
      f32x2_split(rho2, rho_lo, rho_hi);
      f32x2_split(msum2, m_lo, m_hi);
      if (ti >= 2) mbar_wait(&bar_mass_free[par], ((ti >> 1) - 1) & 1, ab, kDqWaitMass);
      s_rho[par][wg][row] = rho_lo + rho_hi;
      s_m[par][wg][row] = m_lo + m_hi;
      mbar_arrive(&bar_mass_ready[par]);
#ifdef GPROJ_TRACE
      if ((threadIdx.x & 127) == 0) tile_event(1 + wg, lin, T, ev_n0, ev_n1, ev_n2, global_ns(), ev_c0, clock64());
#endif
      g0 += T;
    }
  } else {
    // ---------------------------------------------------------------- row constants one tile ahead, and the epilogue: thread <-> query row
    // (keeps the 80 registers of the launch)
    const int ew = warp - C::kDqEpiWarp, row = 32 * ew + lane;
    const uint32_t lane_addr = static_cast<uint32_t>(32 * ew) << 16;
    auto row_constants = [&](int lin, int par) {
      const TileInfo tl = tile_of(lin);
      const int bh = hix(lin);
      const size_t row0 = static_cast<size_t>(bh) * N + tl.row0;
      const float lse_row = (tl.row0 + row < tl.seq_end) ? LSE[row0 + row] : 0.f;
      saved_output_dots<D, 32>(Og + row0 * D, dOg + row0 * D, 32 * ew, tl.seq_end - tl.row0, s_D[par]);
      __syncwarp();
      s_lse[par][row] = lse_row;
      const int rel = tl.row0 + row - tl.seq0;             // row inside the sequence; its last 64-row block is padded with zeros
      if (rank == 0 && rel < ((tl.seq_end - tl.seq0 + 63) / 64) * 64)
        write_row_constants(stats, static_cast<size_t>(bh) * nblk + tl.blk0 + (rel >> 6), rel & 63, -lse_row * 1.4426950408889634f, s_D[par][row], scale_log2);
      mbar_arrive(&bar_stats_ready[par]);
    };
    int ti = 0, lin = sched.next();
    while (lin >= 0) {
      const int next = sched.next(), par = ti & 1;
      // The constants of tile ti + 1 overwrite those of tile ti - 1, whose readers have all handed in their row masses.
      if (!SHORT && next >= 0) row_constants(next, par ^ 1);
      const TileInfo tl = tile_of(lin);
      // q of this warp's 32 rows, D / 8 lanes to a row (whole lines per load and store; one row per thread touches 32
      // lines with every instruction and took 2.2 us instead of 1 us of the tail at d = 128), the first kQ loads ahead of
      // the wait
      constexpr int kCols = D / CL;                        // columns this CTA writes, from col0 on
      constexpr int L = kCols / 8, RPI = 32 / L, kIters = 32 / RPI;
      const int col0 = CL == 1 ? 0 : rank * kCols;
      const int sub = lane / L, part = lane % L;
      const size_t wrow0 = (static_cast<size_t>(hix(lin)) * N + tl.row0 + 32 * ew) * D + col0;
      const int wrows = tl.seq_end - tl.row0 - 32 * ew;    // rows of this warp that exist
      constexpr int kQ = D / CL == 128 ? 8 : 4;            // loads in flight (80 registers at d = 64)
      uint4 qv[kQ];
      auto fetch_q = [&](int h) {
#pragma unroll
        for (int k = 0; k < kQ; ++k) {
          const int r = (kQ * h + k) * RPI + sub;
          qv[k] = r < wrows ? __ldg(reinterpret_cast<const uint4 *>(Qg + wrow0 + static_cast<size_t>(r) * D) + part) : make_uint4(0u, 0u, 0u, 0u);
        }
      };
      fetch_q(0);
      // row masses of all warpgroups (fixed order), lambda = rho / m with the zero-mass rule (Algorithm 1 line 14)
      mbar_wait(&bar_mass_ready[par], (ti >> 1) & 1, ab, kDqWaitMass, kTileBudget);
      float rho_t = s_rho[par][0][row], m_t = s_m[par][0][row];
#pragma unroll
      for (int w = 1; w < C::kWG; ++w) { rho_t += s_rho[par][w][row]; m_t += s_m[par][w][row]; }
      mbar_arrive(&bar_mass_free[par]);
      if (CL > 1) {
        const uint32_t peer = cluster_map_shared(smem_u32(&s_peer[2 * par][row]), rank ^ 1);
        cluster_store_f32(peer, rho_t);
        cluster_store_f32(peer + 512, m_t);
        cluster_mbar_arrive(cluster_map_shared(smem_u32(&bar_peer_mass), rank ^ 1));
        mbar_wait_cluster(&bar_peer_mass, ti & 1, ab, kDqWaitPeer, kTileBudget);
        rho_t += s_peer[2 * par][row];                     // two terms: the same sum in both CTAs
        m_t += s_peer[2 * par + 1][row];
      }
      const float lam = (m_t != 0.f) ? __fdiv_rn(rho_t, m_t) : 0.f;
      const float lam_q = (flags & kFlagNoQCorrection) ? 0.f : lam, lam_k = (flags & kFlagNoKCorrection) ? 0.f : lam;
      // z = BF16(fl32[lambda q]), stored negated (the sign flip is exact), while the last products still run
#pragma unroll
      for (int h = 0; h < kIters / kQ; ++h) {
#pragma unroll
        for (int k = 0; k < kQ; ++k) {
          const int r = (kQ * h + k) * RPI + sub;
          const float lr = __shfl_sync(0xffffffffu, lam_k, r);
          const uint32_t qw[4] = {qv[k].x, qv[k].y, qv[k].z, qv[k].w};
          uint32_t zw[4];
#pragma unroll
          for (int w = 0; w < 4; ++w)
            zw[w] = pack_bf16x2(__fmul_rn(lr, bf16_lo_to_f32(qw[w])), __fmul_rn(lr, bf16_hi_to_f32(qw[w]))) ^ 0x80008000u;
          if (r < wrows) reinterpret_cast<uint4 *>(Zg + wrow0 + static_cast<size_t>(r) * D)[part] = make_uint4(zw[0], zw[1], zw[2], zw[3]);
        }
        if (h + 1 < kIters / kQ) fetch_q(h + 1);
      }
      mbar_wait(&bar_acc_done, ti & 1, ab, kDqWaitAcc, kTileBudget);
      tc_fence_after();
      uint8_t *stg = sStaging + 4096 * ew;
      // The other CTA's parts land in this tile's Q / dO buffer, whose last reader (the last score product) is done:
      // [A, B][kCols / 16 chunks of 16 columns][128 rows] x 64 bytes of FP32, the 16-byte pieces of a row swizzled.
      uint8_t *parts = sRes + (ti % R) * 2 * C::kBigTileBytes;
      auto piece = [&](int chunk, int v) { return static_cast<uint32_t>(chunk * 8192 + row * 64 + ((v ^ ((row >> 1) & 3)) << 4)); };
      if (CL > 1) {
        if (row == 0) cluster_mbar_arrive(cluster_map_shared(smem_u32(&bar_peer_ready), rank ^ 1));
        mbar_wait_cluster(&bar_peer_ready, ti & 1, ab, kDqWaitPeer, kTileBudget);
        const uint32_t peer = cluster_map_shared(smem_u32(parts), rank ^ 1);
#pragma unroll
        for (int c = 0; c < 2 * kCols / 16; ++c) {         // A, then B, of the other CTA's columns
          const int cc = c % (kCols / 16);
          uint32_t a[16];
          tmem_ld16(tmem_base + (c < kCols / 16 ? C::kColAcc0 : C::kColAcc1) + lane_addr + (D - kCols - col0) + 16 * cc, a);
          tmem_wait_ld();
#pragma unroll
          for (int v = 0; v < 4; ++v)
            cluster_store_f4(peer + piece(c, v), __uint_as_float(a[4 * v]), __uint_as_float(a[4 * v + 1]), __uint_as_float(a[4 * v + 2]), __uint_as_float(a[4 * v + 3]));
        }
        cluster_mbar_arrive(cluster_map_shared(smem_u32(&bar_peer_full), rank ^ 1));
        mbar_wait_cluster(&bar_peer_full, ti & 1, ab, kDqWaitPeer, kTileBudget);
      }
      constexpr int kHd = kCols < 64 ? kCols : 64;         // columns staged at a time
#pragma unroll
      for (int hd = 0; hd < kCols / kHd; ++hd) {
#pragma unroll
        for (int cc = 0; cc < kHd / 16; ++cc) {
          uint32_t a[16], b[16];
          tmem_ld16(tmem_base + C::kColAcc0 + lane_addr + col0 + kHd * hd + 16 * cc, a);
          tmem_ld16(tmem_base + C::kColAcc1 + lane_addr + col0 + kHd * hd + 16 * cc, b);
          tmem_wait_ld();
          if (hd == kCols / kHd - 1 && cc == kHd / 16 - 1) { tc_fence_before(); mbar_arrive(&bar_acc_free); }   // the accumulators may be overwritten by the next tile
          if (CL > 1) {
#pragma unroll
            for (int v = 0; v < 4; ++v) {
              const float4 pa = *reinterpret_cast<const float4 *>(parts + piece((kHd / 16) * hd + cc, v)), pb = *reinterpret_cast<const float4 *>(parts + piece(kCols / 16 + (kHd / 16) * hd + cc, v));
              const float fa[4] = {pa.x, pa.y, pa.z, pa.w}, fb[4] = {pb.x, pb.y, pb.z, pb.w};
#pragma unroll
              for (int w = 0; w < 4; ++w) {
                a[4 * v + w] = __float_as_uint(__fadd_rn(__uint_as_float(a[4 * v + w]), fa[w]));
                b[4 * v + w] = __float_as_uint(__fadd_rn(__uint_as_float(b[4 * v + w]), fb[w]));
              }
            }
          }
#pragma unroll
          for (int v = 0; v < 2; ++v) {
            uint32_t dqw[4];
#pragma unroll
            for (int w = 0; w < 4; ++w) {
              const int i = 8 * v + 2 * w;
              const float g0v = __fmul_rn(alpha, __fsub_rn(__uint_as_float(a[i]), __fmul_rn(lam_q, __uint_as_float(b[i]))));
              const float g1v = __fmul_rn(alpha, __fsub_rn(__uint_as_float(a[i + 1]), __fmul_rn(lam_q, __uint_as_float(b[i + 1]))));
              dqw[w] = pack_bf16x2(g0v, g1v);
            }
            *reinterpret_cast<uint4 *>(stg + swz128_offset(lane, 2 * cc + v)) = make_uint4(dqw[0], dqw[1], dqw[2], dqw[3]);
          }
        }
        __syncwarp();
        constexpr int LS = kHd / 8, RS = 32 / LS;          // lanes per row, rows per warp-wide store
#pragma unroll
        for (int k = 0; k < 32 / RS; ++k) {
          const int r = RS * k + lane / LS;
          const uint4 v = *reinterpret_cast<const uint4 *>(stg + swz128_offset(r, lane % LS));
          if (r < wrows) reinterpret_cast<uint4 *>(dQg + wrow0 + static_cast<size_t>(r) * D + kHd * hd)[lane % LS] = v;
        }
        __syncwarp();
      }
      if (CL > 1) {
        fence_proxy_async_smem();
        mbar_arrive(&bar_res_free[ti % R]);                // the parts have been read: the buffer may be loaded again
      }
      lin = next;
      ++ti;
    }
  }

  tc_fence_before();
  if (CL > 1) cluster_sync(); else __syncthreads();   // no CTA leaves while the other one may still write to it
  if (warp == 1) tmem_dealloc(tmem_base, C::kTmemCols);
}

// ============================================================================================
// dK / dV side
// ============================================================================================
// CL = 2: a cluster of two CTAs shares every tile: CTA r takes its steps r, r + 2, ... (over all query heads of the group), then
// CTA 0 gets both parts of dV, CTA 1 both parts of dK, over the consumed K / V tile (its 64 KB hold one 128 x 128 part in
// FP32), added in FP32 before the cast.  Bound where whole tiles are used: the CTA with the longest tile, since a causal or
// grouped call has few tiles of very different length.  This kernel alone, whole tiles -> pairs, d = 128, causal: 16 query / 4 KV
// heads x 4096: 275 -> 151 us (1136 TFLOP/s); 4 heads x 4000: 72.2 -> 53.0; 4 heads x 2048: 43.1 -> 31.3.
template <int D, bool CAUSAL, int CL>
__global__ void __launch_bounds__(BwdCfg<D>::kDkvThreads, 1)
bwd_dkv_kernel(const __grid_constant__ CUtensorMap tmK,    // box 64 x 128 rows
               const __grid_constant__ CUtensorMap tmV,    // box 64 x 128 rows
               const __grid_constant__ CUtensorMap tmQ,    // box 64 x 64 rows
               const __grid_constant__ CUtensorMap tmdO,   // box 64 x 64 rows
               const __grid_constant__ CUtensorMap tmZ,    // box 64 x 64 rows
               const float *__restrict__ stats,
               __nv_bfloat16 *__restrict__ dKg, __nv_bfloat16 *__restrict__ dVg,
               const int4 *__restrict__ plan, int nblk,                           // packed sequences: tile list; statistic blocks per head
               int N, int Nq, int BH, int Hkv, int G, int total_tiles, const ItemOrder order, float scale_log2, float alpha, unsigned flags, int *status) {
  // BH counts (batch, KV head) pairs here.  With grouped queries (G > 1) one work item walks the query steps of all G
  // query heads of its KV head, so their contributions are summed in the FP32 accumulators (Section 3.1: key and value
  // contributions also sum over the query heads that share a KV head).
  using C = BwdCfg<D>;
  constexpr int NB = C::kNB, S = C::kDkvStages;
  extern __shared__ uint8_t smem_raw[];
  uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t *sK = smem;
  uint8_t *sV = sK + C::kBigTileBytes;
  uint8_t *sStage = sV + C::kBigTileBytes;   // stage s: Q, dO, Z step tiles, then the 64-row block of the row-constant tile
  uint8_t *sStaging = sStage + S * C::kDkvStageBytes;   // epilogue warp w: 2048 w

  __shared__ uint64_t bar_res_full, bar_res_free, bar_q_full[S], bar_q_empty[S];
  __shared__ uint64_t bar_s_full[NB], bar_dp_full[NB], bar_r_ready[NB], bar_t_ready[NB], bar_acc_done, bar_acc_free, bar_drain[2], bar_peer_ready, bar_peer_full;
  __shared__ uint32_t tmem_base_smem;
  __shared__ int cta_abort, cta_skip;

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) cta_skip = *reinterpret_cast<volatile int *>(status);
  __syncthreads();
  if (CL == 1 && cta_skip != 0) { griddep_wait(); return; }   // a cluster runs on with every wait falling through: its CTAs exchange results

  const bool use_z = (flags & kFlagNoKCorrection) == 0;
  const uint32_t stage_tx = (use_z ? 3 : 2) * C::kStepTileBytes + kExtBlockBytes;
  // Constant operand of the extra K = 16 slice of the score products: three eight-row core matrices (zeros, rows of
  // (1, 1, 1, 0, 0, 0, 0, 0), zeros).  S^T reads (ones, zeros): it adds columns 0..2 of the row-constant tile, the three
  // BF16 pieces of -LSE / alpha; dP^T reads (zeros, ones): columns 8..10, the pieces of -D.
  __shared__ __align__(128) uint4 s_ones[24];
  if (threadIdx.x < 24) {
    s_ones[threadIdx.x] = (threadIdx.x >= 8 && threadIdx.x < 16) ? make_uint4(0x3f803f80u, 0x00003f80u, 0u, 0u) : make_uint4(0u, 0u, 0u, 0u);
    fence_proxy_async_smem();
  }

  AbortState ab{status, &cta_abort};
  if (threadIdx.x == 0) {
    cta_abort = CL > 1 ? cta_skip : 0;
    mbar_init(&bar_res_full, 1);
    mbar_init(&bar_res_free, CL > 1 ? 1 + 128 : 1);
    for (int s = 0; s < S; ++s) { mbar_init(&bar_q_full[s], 1); mbar_init(&bar_q_empty[s], 1); }
    for (int b = 0; b < NB; ++b) {
      mbar_init(&bar_s_full[b], 1); mbar_init(&bar_dp_full[b], 1);
      mbar_init(&bar_r_ready[b], 128 * C::kSlices); mbar_init(&bar_t_ready[b], 128 * C::kSlices);
    }
    mbar_init(&bar_acc_done, 1);
    mbar_init(&bar_peer_ready, 1);
    mbar_init(&bar_peer_full, 128);
    mbar_init(&bar_acc_free, 128);
    mbar_init(&bar_drain[0], 1);
    mbar_init(&bar_drain[1], 1);
    fence_mbar_init();
  }
  if (warp == 1) { tmem_alloc(&tmem_base_smem, C::kTmemCols); tmem_relinquish(); }
  if (warp == 0 && lane == 0) {
    tma_prefetch_desc(&tmK); tma_prefetch_desc(&tmV); tma_prefetch_desc(&tmQ); tma_prefetch_desc(&tmdO); tma_prefetch_desc(&tmZ);
  }
  tc_fence_before();
  if (CL > 1) cluster_sync(); else __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = __shfl_sync(0xffffffffu, tmem_base_smem, 0);
  griddep_launch_dependents();   // the next kernel in the stream may set itself up beside this one

  TileSched sched(total_tiles, order.solo, CL);
  const int rank = CL > 1 ? cluster_rank() : 0;
  // tile decode: causal -> key tile 0 has the most query steps and comes first
  // Ragged N: query steps round up.  A zero-filled query column past N contributes exactly nothing (its dO, Q and Z rows
  // are zero and its padded statistics are zero, so t = 0 and r multiplies zero rows); key rows past N are clipped on store.
  // In a packed layout the query columns past the end of the sequence are the next sequence's rows and are masked.
  // N: key rows per head (own operand), Nq: query rows per head.  A key j is seen by the queries i >= j - (L_k - L_q).
  auto tix = [&](int lin) { return order.rank(lin); };
  auto hix = [&](int lin) { return order.head(lin); };
  auto tile_of = [&](int lin) { return tile_info(plan, tix(lin), tix(lin), N, Nq); };
  // First query (inside its sequence, rounded down to a 64-row statistics block) that sees this key tile, and the steps
  // from there to the end of the queries; at least one step, fully masked if no query sees the tile.
  auto q_start_of = [&](const TileInfo &t) {
    const int Lq = t.oseq_end - t.oseq0, off = (t.seq_end - t.seq0) - Lq;
    const int first = CAUSAL ? (max(0, t.row0 - t.seq0 - off) & ~63) : 0;
    return min(first, ((Lq - 1) >> 6) << 6);
  };
  auto steps_of = [&](const TileInfo &t) { return max(1, (t.oseq_end - t.oseq0 - q_start_of(t) + C::kStepRows - 1) / C::kStepRows); };
  // This CTA's steps of a tile whose heads have T steps each, and the n-th of them; a CTA that gets none runs step 0 fully
  // masked.
  auto own_steps = [&](int T) { return CL == 1 ? G * T : max(1, (G * T - rank + CL - 1) / CL); };
  auto own_step = [&](int n, int T) { return CL == 1 ? n : (rank < G * T ? CL * n + rank : 0); };
  auto tile_budget = [&]() { return tile_wait_budget(static_cast<long long>(G) * (Nq / C::kStepRows + 1)); };   // of a wait that may span a tile

  if (warp == 0) {
    // ---------------------------------------------------------------- TMA producer of the streamed (Q, dO, Z, stats) step tiles
    if (lane == 0) {
      // Z and the row statistics come from the dQ-side kernel, which may still be running (programmatic dependent
      // launch); everything this CTA did so far, and the stationary-tile loads of the other loader warp, did not need it.
      griddep_wait();
      int g = 0;
      for (int lin = sched.next(); lin >= 0; lin = sched.next()) {
        const TileInfo tl = tile_of(lin);
        const int bh = hix(lin), T = steps_of(tl), q_start = q_start_of(tl);
        const int q_head0 = (bh / Hkv) * (Hkv * G) + (bh % Hkv) * G;     // first query head of the group (flat index)
        for (int m = 0; m < own_steps(T); ++m, ++g) {
          const int st = g % S, n = own_step(m, T);
          if (g >= S) mbar_wait(&bar_q_empty[st], ((g / S) - 1) & 1, ab, kDkvWaitQEmpty);
          mbar_expect_tx(&bar_q_full[st], stage_tx);
          uint8_t *dst = sStage + st * C::kDkvStageBytes;
          const int qh = q_head0 + n / T, qrel = q_start + (n % T) * C::kStepRows, qrow = tl.oseq0 + qrel;
          for (int s = 0; s < C::kSlabs; ++s) {
            tma_load_3d(dst + s * C::kStepSlabBytes, &tmQ, &bar_q_full[st], s * 64, qrow, qh);
            tma_load_3d(dst + C::kStepTileBytes + s * C::kStepSlabBytes, &tmdO, &bar_q_full[st], s * 64, qrow, qh);
            if (use_z) tma_load_3d(dst + 2 * C::kStepTileBytes + s * C::kStepSlabBytes, &tmZ, &bar_q_full[st], s * 64, qrow, qh);
          }
          bulk_load_1d(dst + 3 * C::kStepTileBytes, reinterpret_cast<const uint8_t *>(stats) + (static_cast<size_t>(qh) * nblk + tl.blk0 + (qrel >> 6)) * kExtBlockBytes,
                       kExtBlockBytes, &bar_q_full[st]);
        }
      }
      if (cta_abort) {
        for (int q = (g > S ? g - S : 0); q < g; ++q)
          for (int spin = 0; spin < 100000 && !mbar_try_wait(&bar_q_full[q % S], (q / S) & 1); ++spin) {}
      }
    }
  } else if (warp == 3) {
    // ---------------------------------------------------------------- TMA loader of the stationary (K, V) tiles
    if (lane == 0) {
      int ti = 0;
      for (int lin = sched.next(); lin >= 0; lin = sched.next(), ++ti) {
        const int bh = hix(lin), krow0 = tile_of(lin).row0;
        if (ti >= 1) mbar_wait(&bar_res_free, (ti - 1) & 1, ab, kDkvWaitResFree, tile_budget());
        mbar_expect_tx(&bar_res_full, 2 * C::kBigTileBytes);
        for (int s = 0; s < C::kSlabs; ++s) {
          tma_load_3d(sK + s * C::kBigSlabBytes, &tmK, &bar_res_full, s * 64, krow0, bh);
          tma_load_3d(sV + s * C::kBigSlabBytes, &tmV, &bar_res_full, s * 64, krow0, bh);
        }
      }
      if (cta_abort && ti > 0)
        for (int spin = 0; spin < 100000 && !mbar_try_wait(&bar_res_full, (ti - 1) & 1); ++spin) {}
    }
  } else if (warp == 1) {
    // ---------------------------------------------------------------- tensor-core issuer 1: scores (warp-uniform loop, elected issue)
    constexpr uint32_t idesc_s = idesc_bf16_f32(128, 64, 0, 0);    // [128 keys] x [64 queries], contraction over d
    const SmemDesc dscK = make_smem_desc(smem_u32(sK), 16, 1024), dscV = make_smem_desc(smem_u32(sV), 16, 1024);
    const SmemDesc dscQ0 = make_smem_desc(smem_u32(sStage), 16, 1024);                       // K-major view of stage 0
    const SmemDesc dscOnesS = make_smem_desc_noswizzle(smem_u32(s_ones) + 128, 128, 0);      // (ones, zeros), every row group the same
    const SmemDesc dscOnesP = make_smem_desc_noswizzle(smem_u32(s_ones), 128, 0);            // (zeros, ones)
    const SmemDesc dscExt0 = make_smem_desc_noswizzle(smem_u32(sStage + 3 * C::kStepTileBytes), 128, 256);
    int g = 0, ti = 0;
    for (int lin = sched.next(); lin >= 0; lin = sched.next(), ++ti) {
      const int T = own_steps(steps_of(tile_of(lin)));
      mbar_wait(&bar_res_full, ti & 1, ab, kDkvWaitKV);
      for (int n = 0; n < T; ++n, ++g) {
        const int st = g % S, b = g % NB;
        mbar_wait(&bar_q_full[st], (g / S) & 1, ab, kDkvWaitQ);
        if (g >= NB) mbar_wait(&bar_q_empty[(g - NB) % S], ((g - NB) / S) & 1, ab, kDkvWaitBuf);   // step g - NB done: its r, t are consumed
        tc_fence_after();
        const SmemDesc dscQ = dscQ0.advanced(st * C::kDkvStageBytes), dscdO = dscQ.advanced(C::kStepTileBytes);
        const uint32_t tS = tmem_base + 128 * b, tdP = tS + 64;
        if (elect_one_sync()) {
#pragma unroll
          for (int k = 0; k < D / 16; ++k) {
            const uint32_t oa = (k / 4) * C::kBigSlabBytes + (k % 4) * 32, ob = (k / 4) * C::kStepSlabBytes + (k % 4) * 32;
            umma_ss(tS, dscK.at(oa), dscQ.at(ob), idesc_s, k > 0);
          }
          umma_ss(tS, dscOnesS.at(0), dscExt0.at(st * C::kDkvStageBytes), idesc_s, 1u);     // - LSE / alpha in every key row
          umma_commit(&bar_s_full[b]);                      // phase 1 of the ALUs needs only S^T
#pragma unroll
          for (int k = 0; k < D / 16; ++k) {
            const uint32_t oa = (k / 4) * C::kBigSlabBytes + (k % 4) * 32, ob = (k / 4) * C::kStepSlabBytes + (k % 4) * 32;
            umma_ss(tdP, dscV.at(oa), dscdO.at(ob), idesc_s, k > 0);
          }
          umma_ss(tdP, dscOnesP.at(0), dscExt0.at(st * C::kDkvStageBytes), idesc_s, 1u);    // - D in every key row
          umma_commit(&bar_dp_full[b]);
          if (n == T - 1) umma_commit(&bar_res_free);   // no MMA reads this K / V tile any more
        }
        __syncwarp();
      }
    }
    drain_mmas_if_aborted(&bar_drain[0], ab);
  } else if (warp == 2) {
    // ---------------------------------------------------------------- tensor-core issuer 2: dV += r^T dO, dK += t^T Q + r^T Z
    constexpr uint32_t idesc_a = idesc_bf16_f32(128, D, 0, 1);     // [128 keys] x [d], contraction over 64 queries
    const SmemDesc dscQ0mn = make_smem_desc(smem_u32(sStage), C::kStepSlabBytes, 1024);    // MN-major view of stage 0
    int g = 0, ti = 0;
    for (int lin = sched.next(); lin >= 0; lin = sched.next(), ++ti) {
      const int T = own_steps(steps_of(tile_of(lin)));
      if (ti > 0) mbar_wait(&bar_acc_free, (ti - 1) & 1, ab, kDkvWaitAccFree, tile_budget());   // the previous epilogue has read dV, dK
      for (int p = 0; p < T; ++p, ++g) {
        const int st = g % S, b = g % NB;
        const SmemDesc dscQ = dscQ0mn.advanced(st * C::kDkvStageBytes), dscdO = dscQ.advanced(C::kStepTileBytes),
                       dscZ = dscdO.advanced(C::kStepTileBytes);
        // packed BF16 operands of query slice k (16 queries): r^T over columns 16 k .. 16 k + 7 of the buffer, t^T over the next eight
        const uint32_t tR = tmem_base + 128 * b, tT = tR + 8;
        const uint32_t acc = (p > 0) ? 1u : 0u;
        mbar_wait(&bar_r_ready[b], (g / NB) & 1, ab, kDkvWaitTR);        // r^T is complete: its products run while t^T is computed
        tc_fence_after();
        if (elect_one_sync()) {
#pragma unroll
          for (int k = 0; k < C::kStepRows / 16; ++k)        // dV += r^T dO
            umma_ts(tmem_base + C::kColAcc0, tR + 16 * k, dscdO.at(k * 2048), idesc_a, k > 0 ? 1u : acc);
          if (use_z) {
#pragma unroll
            for (int k = 0; k < C::kStepRows / 16; ++k)      // dK += r^T (-BF16(lambda Q))   (Algorithm 1 lines 17-18)
              umma_ts(tmem_base + C::kColAcc1, tR + 16 * k, dscZ.at(k * 2048), idesc_a, k > 0 ? 1u : acc);
          }
        }
        __syncwarp();
        mbar_wait(&bar_t_ready[b], (g / NB) & 1, ab, kDkvWaitTR);
        tc_fence_after();
        if (elect_one_sync()) {
          const uint32_t acc_k = use_z ? 1u : acc;           // with the correction, dK already holds this step's r^T Z
#pragma unroll
          for (int k = 0; k < C::kStepRows / 16; ++k)        // dK += t^T Q
            umma_ts(tmem_base + C::kColAcc1, tT + 16 * k, dscQ.at(k * 2048), idesc_a, k > 0 ? 1u : acc_k);
          umma_commit(&bar_q_empty[st]);                    // step done: its stage and its score buffer are free
          if (p == T - 1) umma_commit(&bar_acc_done);
        }
        __syncwarp();
      }
    }
    drain_mmas_if_aborted(&bar_drain[1], ab);
  } else if (warp < C::kDkvEpiWarp) {
    // ---------------------------------------------------------------- compute: thread <-> (key row, query slice of every kGroups-th step)
    const int wg = (warp - 4) >> 2, grp = wg / C::kSlices, slice = wg % C::kSlices;
    const int row = 32 * (warp & 3) + lane;                  // key row within the tile
    const uint32_t lane_addr = static_cast<uint32_t>(32 * (warp & 3)) << 16;
    const uint32_t slice_addr = tmem_base + lane_addr + C::kSliceCols * slice;
    int g0 = 0;
    for (int lin = sched.next(); lin >= 0; lin = sched.next()) {
      const TileInfo tl = tile_of(lin);
      const int Th = steps_of(tl), T = own_steps(Th), q_start = q_start_of(tl);
#ifdef GPROJ_TRACE
      const unsigned long long tile_t0 = global_ns();
#endif
      for (int n = (grp - g0 % C::kGroups + C::kGroups) % C::kGroups; n < T; n += C::kGroups) {
        const int g = g0 + n, b = g % NB;
        mbar_wait(&bar_s_full[b], (g / NB) & 1, ab, kDkvWaitSdP);
        tc_fence_after();
        const uint32_t tS16 = slice_addr + 128 * b, tdP16 = tS16 + 64;
        const int nh = own_step(n, Th) % Th;                        // step within the current query head
        const bool none = CL > 1 && rank >= G * Th;                 // a step of the other CTA, run to keep the pipeline in step
        const int Lq = tl.oseq_end - tl.oseq0, off = (tl.seq_end - tl.seq0) - Lq, krel0 = tl.row0 - tl.seq0;
        const int qs = q_start + nh * C::kStepRows;                           // first query (inside its sequence) of the step
        const int q0 = qs + C::kSliceCols * slice;                            // ... of the slice's column 0
        float pkeep[32];
        if ((CAUSAL && qs < krel0 + 128 - off) || qs + C::kStepRows > Lq || none)
          dkv_phase1<true>(tS16, scale_log2, CAUSAL ? krel0 + row - off - q0 : 0, none ? -1 : Lq - 1 - q0, pkeep);
        else
          dkv_phase1<false>(tS16, scale_log2, 0, 0, pkeep);
        tmem_wait_st();
        tc_fence_before();
        mbar_arrive(&bar_r_ready[b]);
        mbar_wait(&bar_dp_full[b], (g / NB) & 1, ab, kDkvWaitSdP);
        tc_fence_after();
        dkv_phase2(tS16, tdP16, pkeep);
        tmem_wait_st();
        tc_fence_before();
        mbar_arrive(&bar_t_ready[b]);
      }

#ifdef GPROJ_TRACE
      if (threadIdx.x == 128) tile_trace(lin, tile_t0, global_ns());
#endif
      g0 += T;
    }
  } else {
    // ---------------------------------------------------------------- epilogue: thread <-> key row.  A finished tile is written out by a
    // warpgroup of its own, so that the compute warpgroups are in the next tile already; it goes through 2 KB of staging
    // per warp (there is no room for a tile next to K / V), which leaves K / V free for the next load at the last score
    // product instead of after the stores.  Measured, this kernel alone, before -> after: 96 heads x 1000 x 128, causal: 86.7
    // -> 81.0 us; 12 packed pairs of 4000 queries and 9000 keys, 12 heads: 68.1 -> 56.7 us; unchanged (1 %) where a CTA
    // walks few long tiles.
    const int ew = warp - C::kDkvEpiWarp;
    const uint32_t lane_addr = static_cast<uint32_t>(32 * ew) << 16;
    uint8_t *stg = sStaging + 2048 * ew;
    int ti = 0;
    for (int lin = sched.next(); lin >= 0; lin = sched.next(), ++ti) {
      const TileInfo tl = tile_of(lin);
      const size_t wrow0 = (static_cast<size_t>(hix(lin)) * N + tl.row0 + 32 * ew) * D;
      const int wrows = tl.seq_end - tl.row0 - 32 * ew;      // rows of this warp that exist
      mbar_wait(&bar_acc_done, ti & 1, ab, kDkvWaitAcc, tile_budget());
      tc_fence_after();
      if (CL > 1) {
        // [D / 16 chunks of 16 columns][128 rows] x 64 bytes of FP32, the 16-byte pieces of a row swizzled
        const int row = 32 * ew + lane;
        auto piece = [&](int chunk, int v) { return static_cast<uint32_t>(chunk * 8192 + row * 64 + ((v ^ ((row >> 1) & 3)) << 4)); };
        const uint32_t t_own = tmem_base + (rank == 0 ? C::kColAcc0 : C::kColAcc1) + lane_addr, t_send = tmem_base + (rank == 0 ? C::kColAcc1 : C::kColAcc0) + lane_addr;
        const uint32_t peer = cluster_map_shared(smem_u32(sK), rank ^ 1);
        const float scale = rank == 0 ? 1.0f : alpha;
        if (row == 0) cluster_mbar_arrive(cluster_map_shared(smem_u32(&bar_peer_ready), rank ^ 1));   // this CTA's K / V tile is consumed
        mbar_wait_cluster(&bar_peer_ready, ti & 1, ab, kDkvWaitPeer, tile_budget());
#pragma unroll 2
        for (int cc = 0; cc < D / 16; ++cc) {
          uint32_t a[16];
          tmem_ld16(t_send + 16 * cc, a);
          tmem_wait_ld();
#pragma unroll
          for (int v = 0; v < 4; ++v)
            cluster_store_f4(peer + piece(cc, v), __uint_as_float(a[4 * v]), __uint_as_float(a[4 * v + 1]), __uint_as_float(a[4 * v + 2]), __uint_as_float(a[4 * v + 3]));
        }
        cluster_mbar_arrive(cluster_map_shared(smem_u32(&bar_peer_full), rank ^ 1));
        mbar_wait_cluster(&bar_peer_full, ti & 1, ab, kDkvWaitPeer, tile_budget());
#pragma unroll 1
        for (int c = 0; c < D / 32; ++c) {
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            const int cc = 2 * c + h;
            uint32_t a[16], w8[8];
            tmem_ld16(t_own + 16 * cc, a);
            float b[16];
#pragma unroll
            for (int v = 0; v < 4; ++v) *reinterpret_cast<float4 *>(&b[4 * v]) = *reinterpret_cast<const float4 *>(sK + piece(cc, v));
            tmem_wait_ld();
            if (cc == D / 16 - 1) { tc_fence_before(); mbar_arrive(&bar_acc_free); }   // the accumulators may be overwritten by the next tile
#pragma unroll
            for (int i = 0; i < 8; ++i)
              w8[i] = pack_bf16x2(__fmul_rn(scale, __fadd_rn(__uint_as_float(a[2 * i]), b[2 * i])), __fmul_rn(scale, __fadd_rn(__uint_as_float(a[2 * i + 1]), b[2 * i + 1])));
#pragma unroll
            for (int v = 0; v < 2; ++v)
              *reinterpret_cast<uint4 *>(stg + lane * 64 + (((2 * h + v) ^ ((lane >> 1) & 3)) << 4)) = make_uint4(w8[4 * v], w8[4 * v + 1], w8[4 * v + 2], w8[4 * v + 3]);
          }
          __syncwarp();
          __nv_bfloat16 *dst = (rank == 0 ? dVg : dKg) + wrow0 + 32 * c;
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            const int r = 8 * k + (lane >> 2), p = lane & 3;
            const uint4 v = *reinterpret_cast<const uint4 *>(stg + r * 64 + ((p ^ ((r >> 1) & 3)) << 4));
            if (r < wrows) reinterpret_cast<uint4 *>(dst + static_cast<size_t>(r) * D)[p] = v;
          }
          __syncwarp();
        }
        fence_proxy_async_smem();
        mbar_arrive(&bar_res_free);                          // the parts have been read: K and V may be loaded again
        continue;
      }
#pragma unroll 1
      for (int c = 0; c < 2 * D / 32; ++c) {                 // 32-column chunks of dV, then of dK (adjacent accumulator columns)
        const float scale = c < D / 32 ? 1.0f : alpha;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          uint32_t a[16];
          tmem_ld16(tmem_base + C::kColAcc0 + lane_addr + 32 * c + 16 * h, a);
          tmem_wait_ld();
          if (c == 2 * D / 32 - 1 && h == 1) { tc_fence_before(); mbar_arrive(&bar_acc_free); }   // the accumulators may be overwritten by the next tile
#pragma unroll
          for (int v = 0; v < 2; ++v) {
            uint32_t w4[4];
#pragma unroll
            for (int w = 0; w < 4; ++w)
              w4[w] = pack_bf16x2(__fmul_rn(scale, __uint_as_float(a[8 * v + 2 * w])), __fmul_rn(scale, __uint_as_float(a[8 * v + 2 * w + 1])));
            *reinterpret_cast<uint4 *>(stg + lane * 64 + (((2 * h + v) ^ ((lane >> 1) & 3)) << 4)) = make_uint4(w4[0], w4[1], w4[2], w4[3]);
          }
        }
        __syncwarp();
        __nv_bfloat16 *dst = (c < D / 32 ? dVg : dKg) + wrow0 + 32 * (c % (D / 32));
#pragma unroll
        for (int k = 0; k < 4; ++k) {                        // four lanes to a row's 64 bytes
          const int r = 8 * k + (lane >> 2), p = lane & 3;
          const uint4 v = *reinterpret_cast<const uint4 *>(stg + r * 64 + ((p ^ ((r >> 1) & 3)) << 4));
          if (r < wrows) reinterpret_cast<uint4 *>(dst + static_cast<size_t>(r) * D)[p] = v;
        }
        __syncwarp();
      }
    }
  }

  tc_fence_before();
  if (CL > 1) cluster_sync(); else __syncthreads();   // no CTA leaves while the other one may still write to it
  if (warp == 1) tmem_dealloc(tmem_base, C::kTmemCols);
}

}  // namespace gproj
