// Fused attention forward for sm_100a, head dimension 64: three softmax warpgroups on 64-key steps.
//
// Same results as attn_fwd.cuh (subtract-before-scale online softmax on the unscaled logits, lazy running maximum, FP32
// normaliser and accumulator, BF16 probabilities); another pipeline.  One work item is one 128-row query tile.  Its 64-key
// steps are dealt in turn to three softmax warpgroups, each with its own running maximum, normaliser and accumulator, and one
// of them merges the three parts at the end.  Steps are numbered through all items of a CTA; step n belongs to warpgroup n mod 3.
//
// TMEM: five buffers of 64 columns, step n's scores and over them its packed probabilities in buffer n mod 5, and O_w at 320 + 64 w
// (w = 0..2).  The scores of step n + 3 are computed while the warpgroup is in step n, and nobody but the tensor core waits for
// a product P~V (except to rescale O_w, which is rare, and at the end of an item).
//
// What bounds it.  The exponentials of a key tile (128 x 128) keep the special-function unit busy for 1024 clk; with all that goes
// with them (maximum, subtraction, scale, sum, packing, TMEM) two or more warps per scheduler sustain 1140.  Each warp also spends
// 700 to 1000 clk per step on barriers, TMEM loads and the maximum, in which the others have the unit to themselves: with two
// warps per scheduler it idled a third of the time, and throughout an item's epilogue (its pipe over a launch of 16 heads x 4096, by ncu:
// 59 % of the peak then, 65 % now).  Three warps per scheduler
// hide that better (more than three do not fit: 64 columns of TMEM for each O_w and at least 64 for its scores), the
// merge of an item runs in one warpgroup while the others are in the next, and short items cost a third of what they did.
// Measured, forward alone, two warpgroups on 128 keys (pairs or split tiles) -> this: 16 heads x 4096, causal: 58.0 -> 51.5 us; 96 x
// 1000: 35.5 -> 29.8; 32 x 8192: 422 -> 391; 24 packed documents, 16676 rows, 16 heads: 101.8 -> 78.1; 200 documents of 30 to 300
// rows: 178.8 -> 113.8; 64 x 2000, not causal: 117.6 -> 92.9; 32 x 8192, not causal: 730 -> 677.
// Tried: four warpgroups with P~_w over S_w (59 us on the first of these; each product P~V is then on its warpgroup's way), P~_w
// apart from S_w (55; waits for P~V), a pool for the probabilities alone (57.5), P~V(n) and S(n + 5) from one thread (63).
#pragma once
#include "attn_fwd.cuh"

namespace gproj {

struct FwdW64Cfg {
  static constexpr int D = 64;
  static constexpr int kBlockM = 128, kStep = 64;
  static constexpr int kWG = 3;
  static constexpr int kQBytes = 128 * 128, kStepBytes = 64 * 128;
  static constexpr int kQBufs = 3;
  static constexpr int kStages = 8;                        // ring of (K, V) step tiles
  static constexpr int kStageBytes = 2 * kStepBytes;
  static constexpr int kSmemBytes = kQBufs * kQBytes + kStages * kStageBytes + 1024;
  static constexpr int kThreads = 128 + 128 * kWG;
  static constexpr int kRegsSoftmax = 144, kRegsAux = 80;  // of 512 x 128 at launch
  static_assert(kWG * kRegsSoftmax + kRegsAux <= 4 * 128, "register shares");
  static constexpr int kTmemCols = 512;
  static constexpr int kBufs = 5;
  static constexpr uint32_t kColO = 64 * kBufs;
  static_assert(64 * (kBufs + kWG) <= kTmemCols, "TMEM budget");
};

// z = exp2(..) of the 64 columns of one row, as softmax_exp_store.
template <bool FMA_SOFTMAX>
__device__ __forceinline__ float softmax_exp_store64(const uint32_t (&xr)[2][32], uint32_t tP, float m_new, float scale_log2, float m_scaled) {
  const uint64_t negm2 = f32x2(-m_new, -m_new), scale2 = f32x2(scale_log2, scale_log2), negms2 = f32x2(-m_scaled, -m_scaled);
  uint64_t rs2[2] = {f32x2(0.f, 0.f), f32x2(0.f, 0.f)};
#pragma unroll
  for (int c = 0; c < 2; ++c) {
    uint32_t pk[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) {
      const uint64_t x2 = f32x2_bits(xr[c][2 * i], xr[c][2 * i + 1]);
      const uint64_t a2 = FMA_SOFTMAX ? fma2(x2, scale2, negms2) : mul2(add2(x2, negm2), scale2);
      float a0, a1;
      f32x2_split(a2, a0, a1);
      const float z0 = fast_exp2(a0), z1 = fast_exp2(a1);
      rs2[i & 1] = add2(rs2[i & 1], f32x2(z0, z1));
      pk[i] = pack_bf16x2(z0, z1);
    }
    tmem_st16(tP + 16 * c, pk);
  }
  float r0, r1, r2, r3;
  f32x2_split(rs2[0], r0, r1);
  f32x2_split(rs2[1], r2, r3);
  return (r0 + r1) + (r2 + r3);
}

template <bool CAUSAL, bool FMA_SOFTMAX>
__global__ void __launch_bounds__(FwdW64Cfg::kThreads, 1)
attn_fwd_w64_kernel(const __grid_constant__ CUtensorMap tmQ,    // box 64 x 128 rows
                    const __grid_constant__ CUtensorMap tmK,    // box 64 x 64 rows
                    const __grid_constant__ CUtensorMap tmV,    // box 64 x 64 rows
                    const __grid_constant__ CUtensorMap tmO,    // store, box 64 x 32 rows
                    __nv_bfloat16 *__restrict__ Og, const int4 *__restrict__ plan, float *__restrict__ LSE, int N, int Nk, int Hq, int G,
                    int total_items, const ItemOrder order, float scale_log2, float alpha, int *status) {
  using C = FwdW64Cfg;
  constexpr int S = C::kStages, R = C::kQBufs, W = C::kWG, NB = C::kBufs;
  extern __shared__ uint8_t smem_raw[];
  uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t *sQ = smem;                               // buffer b: Q tile of items b mod R (later reused to stage O)
  uint8_t *sKV = sQ + R * C::kQBytes;               // stage n mod S: K, then V of step n

  __shared__ uint64_t bar_q_full[R], bar_q_free[R], bar_kv_full[S], bar_kv_empty[S];
  __shared__ uint64_t bar_s_full[NB], bar_p_ready[NB], bar_merge[2], bar_o_free[2], bar_drain[2];
  __shared__ int s_item[2 * R][2];                  // rank and head of an item, from the Q loader to the softmax warps
  __shared__ float s_m[2][W][128], s_l[2][W][128];  // running maximum and normaliser of each part, by item parity
  __shared__ uint32_t tmem_base_smem;
  __shared__ int cta_abort, cta_skip;

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) cta_skip = *reinterpret_cast<volatile int *>(status);
  __syncthreads();

  const int n_qt = (N + C::kBlockM - 1) / C::kBlockM;
  AbortState ab{status, &cta_abort};
  if (threadIdx.x == 0) {
    cta_abort = 0;
    for (auto &slot : s_item) slot[0] = slot[1] = 0;   // see attn_fwd.cuh
    for (int b = 0; b < R; ++b) { mbar_init(&bar_q_full[b], 1); mbar_init(&bar_q_free[b], 4); }
    for (int s = 0; s < S; ++s) { mbar_init(&bar_kv_full[s], 1); mbar_init(&bar_kv_empty[s], 1); }
    for (int b = 0; b < NB; ++b) { mbar_init(&bar_s_full[b], 1); mbar_init(&bar_p_ready[b], 4); }
    for (int p = 0; p < 2; ++p) { mbar_init(&bar_merge[p], 4 * W); mbar_init(&bar_o_free[p], 4); mbar_init(&bar_drain[p], 1); }
    fence_mbar_init();
  }
  if (warp == 1) { tmem_alloc(&tmem_base_smem, C::kTmemCols); tmem_relinquish(); }
  if (warp == 0 && lane == 0) { tma_prefetch_desc(&tmQ); tma_prefetch_desc(&tmK); tma_prefetch_desc(&tmV); tma_prefetch_desc(&tmO); }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = __shfl_sync(0xffffffffu, tmem_base_smem, 0);   // the shuffle marks it warp-uniform

  // Everything so far may have run beside the kernel before this one in the stream; its memory is visible from here on.
  griddep_wait();
  griddep_launch_dependents();
  if (cta_skip != 0) {       // an earlier wait gave up: drain the rest of the grid quickly, but not past the kernel before this one
    __syncthreads();
    if (warp == 1) tmem_dealloc(tmem_base, C::kTmemCols);
    return;
  }

  // Items as in attn_fwd.cuh.  T: 64-key steps up to the last key the tile's last row sees; at least one.
  struct Item { int seq0, len, qt, T, kseq0, klen, off; };
  auto decode_rank = [&](int rank) {
    Item it;
    if (plan != nullptr) {
      const TileInfo ti = tile_info(plan, rank, 0, N, Nk);
      it.seq0 = ti.seq0; it.len = ti.seq_end - ti.seq0; it.qt = (ti.row0 - ti.seq0) / C::kBlockM;
      it.kseq0 = ti.oseq0; it.klen = ti.oseq_end - ti.oseq0;
    } else {
      it.seq0 = 0; it.len = N; it.qt = CAUSAL ? (n_qt - 1 - rank) : rank;
      it.kseq0 = 0; it.klen = Nk;
    }
    it.off = it.klen - it.len;
    const int kend = CAUSAL ? min(it.klen, (it.qt + 1) * C::kBlockM + it.off) : it.klen;
    it.T = max(1, (max(kend, 0) + C::kStep - 1) / C::kStep);
    return it;
  };
  TileSched sched(total_items, order.solo, 1);

  if (warp < 4) {
  setmaxnreg_dec<C::kRegsAux>();
  if (warp == 0) {
    // ---------------------------------------------------------------- TMA producer of the (K, V) step tiles
    if (lane == 0) {
      int n = 0;
      for (int lin = sched.next(); lin >= 0; lin = sched.next()) {
        const Item it = decode_rank(order.rank(lin));
        const int kvh = kv_head_of(order.head(lin), Hq, G);       // grouped-query: the group's shared K / V head
        for (int j = 0; j < it.T; ++j, ++n) {
          const int st = n % S;
          if (n >= S) mbar_wait(&bar_kv_empty[st], ((n / S) - 1) & 1, ab, kFwdWaitKVEmpty);
          uint8_t *dst = sKV + st * C::kStageBytes;
          mbar_expect_tx(&bar_kv_full[st], C::kStageBytes);
          tma_load_3d(dst, &tmK, &bar_kv_full[st], 0, it.kseq0 + j * C::kStep, kvh);
          tma_load_3d(dst + C::kStepBytes, &tmV, &bar_kv_full[st], 0, it.kseq0 + j * C::kStep, kvh);
        }
      }
      if (cta_abort)
        for (int q = (n > S ? n - S : 0); q < n; ++q)
          for (int spin = 0; spin < 100000 && !mbar_try_wait(&bar_kv_full[q % S], (q / S) & 1); ++spin) {}
    }
  } else if (warp == 3) {
    // ---------------------------------------------------------------- TMA loader of the Q tiles
    if (lane == 0) {
      int ti = 0;
      for (int lin = sched.next(); lin >= 0; lin = sched.next(), ++ti) {
        const int rank = order.rank(lin), bh = order.head(lin), qb = ti % R;
        const Item it = decode_rank(rank);
        if (ti >= R) mbar_wait(&bar_q_free[qb], ((ti / R) - 1) & 1, ab, kFwdWaitQFree, tile_wait_budget(2LL * (Nk / C::kStep + 1)));
        s_item[ti % (2 * R)][0] = rank;              // for the softmax warps; the barrier's completion publishes the two words
        s_item[ti % (2 * R)][1] = bh;
        mbar_expect_tx(&bar_q_full[qb], C::kQBytes);
        tma_load_3d(sQ + qb * C::kQBytes, &tmQ, &bar_q_full[qb], 0, it.seq0 + it.qt * C::kBlockM, bh);
      }
      if (cta_abort)
        for (int q = (ti > R ? ti - R : 0); q < ti; ++q)
          for (int spin = 0; spin < 100000 && !mbar_try_wait(&bar_q_full[q % R], (q / R) & 1); ++spin) {}
    }
  } else if (warp == 1) {
    // ---------------------------------------------------------------- tensor-core issuer 1: S_w = Q K(n)^T
    constexpr uint32_t idesc_s = idesc_bf16_f32(128, C::kStep, 0, 0);          // both operands K-major
    const SmemDesc dscQ0 = make_smem_desc(smem_u32(sQ), 16, 1024), dscK0 = make_smem_desc(smem_u32(sKV), 16, 1024);
    // Few instructions to a step: the compute warps of this scheduler leave few issue slots, and the loop's latency is part of the pipeline's.
    // (A wait for the phase before a barrier's first returns at once: e, e_ph start five steps back.)
    uint32_t st = 0, st_ph = 0, b = 0, e = (S - NB) % S, e_ph = 1;
    int ti = 0;
    for (int lin = sched.next(); lin >= 0; lin = sched.next(), ++ti) {
      const int T = decode_rank(order.rank(lin)).T, qb = ti % R;
      mbar_wait(&bar_q_full[qb], (ti / R) & 1, ab, kFwdWaitQ);
      const SmemDesc dscQ = dscQ0.advanced(qb * C::kQBytes);
      for (int j = 0; j < T; ++j) {
        mbar_wait(&bar_kv_full[st], st_ph, ab, kFwdWaitK);
        mbar_wait(&bar_kv_empty[e], e_ph, ab, kFwdWaitSFree);      // the probabilities of step n - NB are consumed
        tc_fence_after();
        const SmemDesc dscK = dscK0.advanced(st * C::kStageBytes);
        if (elect_one_sync()) {
#pragma unroll
          for (int k = 0; k < C::D / 16; ++k) umma_ss(tmem_base + 64 * b, dscQ.at(k * 32), dscK.at(k * 32), idesc_s, k > 0);
          umma_commit(&bar_s_full[b]);
        }
        __syncwarp();
        if (++st == S) { st = 0; st_ph ^= 1; }
        if (++e == S) { e = 0; e_ph ^= 1; }
        if (++b == NB) b = 0;
      }
    }
    drain_mmas_if_aborted(&bar_drain[0], ab);
  } else {
    // ---------------------------------------------------------------- tensor-core issuer 2: O_w += P~_w V(n)
    constexpr uint32_t idesc_o = idesc_bf16_f32(128, C::D, 0, 1);              // V is MN-major
    const SmemDesc dscV0 = make_smem_desc(smem_u32(sKV + C::kStepBytes), C::kStepBytes, 1024);
    uint32_t st = 0, w = 0, b = 0, b_ph = 0;
    int ti = 0;
    for (int lin = sched.next(); lin >= 0; lin = sched.next(), ++ti) {
      const int T = decode_rank(order.rank(lin)).T;
      if (ti > 0) mbar_wait(&bar_o_free[(ti - 1) & 1], ((ti - 1) >> 1) & 1, ab, kFwdWaitOFree);   // the previous item has been merged
      for (int j = 0; j < T; ++j) {
        const SmemDesc dscV = dscV0.advanced(st * C::kStageBytes);
        const uint32_t acc = j >= W ? 1u : 0u, tP = tmem_base + 64 * b, tO = tmem_base + C::kColO + 64 * w;
        mbar_wait(&bar_p_ready[b], b_ph, ab, kFwdWaitP);           // the step's V landed with its K
        tc_fence_after();
        if (elect_one_sync()) {
#pragma unroll
          for (int k = 0; k < C::kStep / 16; ++k) umma_ts(tO, tP + 8 * k, dscV.at(k * 2048), idesc_o, k > 0 ? 1u : acc);
          umma_commit(&bar_kv_empty[st]);                 // step done: its stage and its buffer are free
        }
        __syncwarp();
        if (++st == S) st = 0;
        if (++w == W) w = 0;
        if (++b == NB) { b = 0; b_ph ^= 1; }
      }
    }
    drain_mmas_if_aborted(&bar_drain[1], ab);
  }
  } else {
    // ---------------------------------------------------------------- softmax: thread <-> row of the item's query tile
    setmaxnreg_inc<C::kRegsSoftmax>();
    const int w = (warp - 4) >> 2;
    const int row = 32 * (warp & 3) + lane;
    const uint32_t lane_addr = static_cast<uint32_t>(32 * (warp & 3)) << 16;
    const uint32_t tO = tmem_base + lane_addr + C::kColO + 64 * w;
    int g0 = 0, n = w;         // CTA's steps before this item, this warpgroup's next step
    int b = w, b_ph = 0;       // ... its buffer (n mod NB) and the parity of n / NB
    static_assert(W <= NB && NB < 2 * W, "a step on, the buffer wraps at most once");
    int stored = -1;           // lane 0: Q buffer out of which a tile is being stored
    int ti = 0;
    for (int lin = sched.next(); lin >= 0; lin = sched.next(), ++ti) {
      const int qb = ti % R, par = ti & 1;
      mbar_wait(&bar_q_full[qb], (ti / R) & 1, ab, kFwdWaitQ);     // the item's description has been published
      const Item it = decode_rank(s_item[ti % (2 * R)][0]);
      const int T = it.T, part = (w + W - g0 % W) % W;             // this warpgroup takes steps part, part + W, ...
      const int qrow = it.qt * C::kBlockM + row;
      const int rk = CAUSAL ? min(qrow + it.off, it.klen - 1) : it.klen - 1;                                    // last key of this row
      const int jm = CAUSAL ? min((it.qt * C::kBlockM + it.off + 1) >> 6, it.klen >> 6) : (it.klen >> 6);       // first step that needs the mask
      float m_run = -INFINITY, l_run = 0.f;
      for (int j = part; j < T; j += W) {
        const uint32_t tS = tmem_base + lane_addr + 64 * b;
        mbar_wait(&bar_s_full[b], b_ph, ab, kFwdWaitS);
        tc_fence_after();
        uint32_t xr[2][32];
        tmem_ld32(tS, xr[0]);
        tmem_ld32(tS + 32, xr[1]);
        tmem_wait_ld();
        if (j >= jm) {
          const int lim = rk - j * C::kStep;
#pragma unroll
          for (int c = 0; c < 2; ++c)
#pragma unroll
            for (int i = 0; i < 32; ++i)
              if (32 * c + i > lim) xr[c][i] = 0xff800000u;
        }
        float mxp[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) mxp[i] = fmaxf(__uint_as_float(xr[0][i]), __uint_as_float(xr[0][8 + i]));
#pragma unroll
        for (int e = 16; e < 64; e += 16)
#pragma unroll
          for (int i = 0; i < 8; ++i)
            mxp[i] = fmax3(mxp[i], __uint_as_float(xr[(e + i) >> 5][(e + i) & 31]), __uint_as_float(xr[(e + 8 + i) >> 5][(e + 8 + i) & 31]));
        const float mx = fmax3(fmax3(mxp[0], mxp[1], mxp[2]), fmax3(mxp[3], mxp[4], mxp[5]), fmax3(mxp[6], mxp[7], kFwdMaxFloor));
        float m_new = fmaxf(m_run, mx);
#ifndef GPROJ_FWD_EAGER_MAX
        if (!FMA_SOFTMAX && __fmul_rn(__fsub_rn(m_new, m_run), scale_log2) <= 8.0f) m_new = m_run;
#endif
        const float corr = fast_exp2(__fmul_rn(__fsub_rn(m_run, m_new), scale_log2));
        const float m_scaled = __fmul_rn(m_new, scale_log2);
        const float rs = softmax_exp_store64<FMA_SOFTMAX>(xr, tS, m_new, scale_log2, m_scaled);
        l_run = l_run * corr + rs;
        if (j >= W && __any_sync(0xffffffffu, m_new != m_run)) {
          mbar_wait(&bar_kv_empty[(n - W) % S], ((n - W) / S) & 1, ab, kFwdWaitPV);      // O_w holds all steps before this one
          tc_fence_after();
#pragma unroll
          for (int c = 0; c < 2; ++c) {
            uint32_t o[32];
            tmem_ld32(tO + 32 * c, o);
            tmem_wait_ld();
#pragma unroll
            for (int i = 0; i < 32; ++i) o[i] = __float_as_uint(__uint_as_float(o[i]) * corr);
            tmem_st32(tO + 32 * c, o);
          }
        }
        m_run = m_new;
        tmem_wait_st();
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&bar_p_ready[b]);
        n += W;
        b += W;
        if (b >= NB) { b -= NB; b_ph ^= 1; }
      }
      if (part < T) {
        // this part is complete: leave its statistics for the warpgroup that merges
        mbar_wait(&bar_kv_empty[(n - W) % S], ((n - W) / S) & 1, ab, kFwdWaitPV);
        s_m[par][w][row] = m_run;
        s_l[par][w][row] = l_run;
      }
      const bool merger = (g0 + T - 1) % W == w;                   // the warpgroup with the item's last step
      __syncwarp();
      if (lane == 0) mbar_arrive(&bar_merge[par]);
      // The last tile's buffer is handed back only here: waiting for its store right away kept this item's merge waiting for this warp.
      // Measured, a store of the whole tile waited for at once -> stores by warps, handed back here: 96 heads x 1000: 29.9 -> 28.8 us, 1000 x
      // 64: 15.2 -> 14.3, 16 x 4096: 51.6 -> 51.1, 32 x 4096, not causal: 175.9 -> 172.6; 100 x 128 behind 1000 (one item per CTA): 11.1 -> 11.3.
      if (stored >= 0) {
        bulk_wait_group_read0();
        mbar_arrive(&bar_q_free[stored]);
        stored = -1;
      }
      if (merger) {
        // O = sum_p O_p s_p / L with s_p = exp2((m_p - M) alpha log2 e), in the order of the parts' first keys
        mbar_wait(&bar_merge[par], (ti >> 1) & 1, ab, kFwdWaitMerge);
        tc_fence_after();
        const int bh = s_item[ti % (2 * R)][1], np = min(T, W);
        float a[W], M = kFwdMaxFloor, L = 0.f;
#pragma unroll
        for (int p = 0; p < W; ++p) {
          a[p] = p < np ? s_m[par][(g0 + p) % W][row] : kFwdMaxFloor;
          M = fmaxf(M, a[p]);
        }
#pragma unroll
        for (int p = 0; p < W; ++p) {
          a[p] = fast_exp2(__fmul_rn(__fsub_rn(a[p], M), scale_log2));
          if (p < np) L = fmaf(s_l[par][(g0 + p) % W][row], a[p], L);
        }
        const float inv = (L > 0.f) ? 1.0f / L : 0.f;              // a row with an empty support has l = 0: O = 0
        uint8_t *stage = sQ + qb * C::kQBytes;                     // no product reads this Q tile any more
        const uint32_t tOl = tmem_base + lane_addr + C::kColO;
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          float acc[16];
#pragma unroll
          for (int i = 0; i < 16; ++i) acc[i] = 0.f;
#pragma unroll
          for (int p = 0; p < W; ++p)
            if (p < np) {
              uint32_t o[16];
              tmem_ld16(tOl + 64 * ((g0 + p) % W) + 16 * c, o);
              tmem_wait_ld();
#pragma unroll
              for (int i = 0; i < 16; ++i) acc[i] = fmaf(__uint_as_float(o[i]), a[p], acc[i]);
            }
#pragma unroll
          for (int v = 0; v < 2; ++v) {
            uint32_t pk[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) pk[i] = pack_bf16x2(acc[8 * v + 2 * i] * inv, acc[8 * v + 2 * i + 1] * inv);
            *reinterpret_cast<uint4 *>(stage + swz128_offset(row, 2 * c + v)) = make_uint4(pk[0], pk[1], pk[2], pk[3]);
          }
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&bar_o_free[par]);              // the accumulators may be overwritten by the next item
        const int qrow0 = it.seq0 + it.qt * C::kBlockM;
        if (qrow < it.len) LSE[static_cast<size_t>(bh) * N + qrow0 + row] = (L > 0.f) ? fmaf(M, alpha, logf(L)) : INFINITY;
        const TileInfo tinfo{qrow0, it.seq0, it.seq0 + it.len, 0, 0, 0};
        fence_proxy_async_smem();
        warp_bar_sync(warp);                                       // see there: more than __syncwarp
        if (tile_store_by_tma(tinfo, N)) {                         // by each warp for itself: see attn_fwd.cuh
          if (lane == 0) {
            if (qrow < it.len) tma_store_3d(&tmO, stage + row * 128, 0, qrow0 + row, bh);
            bulk_commit_group();
            stored = qb;
          }
        } else {
          // ragged last tile of a packed sequence that another sequence follows: rows past its end are not ours to write
          store_rows_clipped<C::D>(stage, C::kQBytes, Og + (static_cast<size_t>(bh) * N + qrow0) * C::D, row, it.len - it.qt * C::kBlockM);
          warp_bar_sync(warp);
          if (lane == 0) mbar_arrive(&bar_q_free[qb]);
        }
      }
      g0 += T;
    }
    if (stored >= 0) bulk_wait_group_read0();
  }

  tc_fence_before();
  __syncthreads();
  if (warp == 1) tmem_dealloc(tmem_base, C::kTmemCols);
}

}  // namespace gproj
