// Fused attention forward for sm_100a: O = softmax(alpha Q K^T) V and the row log-sum-exp.
//
// A persistent CTA (one per SM) walks a static list of work items.  Roles (384 threads):
//   warp 0        TMA producer of the streamed K_j / V_j tiles (separate barriers: S needs only K, P~V only V)
//   warp 1        tensor-core issuer 1: S_t = Q K_j^T (N = 128, FP32 in TMEM); owns TMEM
//   warp 2        tensor-core issuer 2: O_t += P~_t V_j with the BF16 probabilities read straight from TMEM
//   warp 3        TMA loader of the stationary Q tile(s)
//   warps 4..7    softmax warpgroup 0, warps 8..11 softmax warpgroup 1: thread <-> query row (TMEM lane), so every
//                 row statistic is a private register.  While one warpgroup is in the ALUs the tensor core works for
//                 the other one (the tensor-core queue is only 1-2 instructions deep, hence two issuing warps: each
//                 one's barrier polls overlap the other's MMAs).
// Work items (template parameter MODE):
//   pairs (5)     one item = two 128-row query tiles of one (batch, head), warpgroup t <-> tile t, every K / V tile
//                 serves both; separate rings for K and V.
//   one tile (0)  the same with one ring, for heads of a single tile, of which there are many: the second warpgroup idles.
//   split (2)     one item = one query tile; warpgroup t takes the key tiles j = t (mod 2) with its own running
//                 maximum, normaliser and accumulator, and warpgroup 0 merges the two halves at the end.  Used when
//                 pairs would leave SMs idle and for packed sequences.
//   split (4)     the same with separate rings for K and V (d = 128, long key ranges).
//   cluster (3)   one item = one query tile on a cluster of 2, 4 or 8 CTAs that share its key tiles in the same way and
//                 merge 4, 8 or 16 parts through distributed shared memory.  Used when even single tiles leave SMs
//                 idle: a block of new queries behind a key history, a short batch.
//   cluster (6)   the same with separate rings for K and V (d = 128, four or more key tiles to a CTA).
// Softmax arithmetic (FMA_SOFTMAX = false, the default): online softmax on the UNSCALED logits with the
// subtract-before-scale rounding of
// Eq. "gproj-forward": z = exp2(fl32[ fl32(x - x_max) * (alpha log2 e) ]); l accumulates the FP32 z, the value
// product uses BF16(z); the running maximum is raised lazily and the accumulator rescaled only then.
// The saved state is BF16 O (staged in the TMA layout over the consumed Q tile, written by a TMA store) and
// FP32 LSE = alpha x_max + ln l  (Algorithm 1, "Input").
// TMEM: see FwdTmem.
#pragma once
#include "attn_bwd.cuh"   // TileSched
#include "sm100_primitives.cuh"

namespace gproj {

// Floor of the running row maximum (see the softmax loop): far below any score, far above -FLT_MAX.
constexpr float kFwdMaxFloor = -1.0e30f;

template <int D>
struct FwdCfg {
  static constexpr int kBlockM = 128;                  // rows of one query tile (two per work item)
  static constexpr int kBlockN = 128;
  static constexpr int kSlabs = D / 64;                // 64-column (128-byte) swizzle slabs per tile
  static constexpr int kSlabBytes = 128 * 128;         // 128 rows x 128 B
  static constexpr int kTileBytes = kSlabs * kSlabBytes;
  static constexpr int kStages = (D == 64) ? 4 : 2;    // ring of (K, V) tile pairs
  static constexpr int kSmemBytes = 2 * kTileBytes + kStages * 2 * kTileBytes + 1024;
  static constexpr int kTmemCols = 512;
  static constexpr uint32_t kColS = 0, kColO = 256;    // O_t at 256 + D t; S_t and P~_t as in FwdTmem
  static constexpr int kThreads = 384;
  // MODE 4, 5 and 6 re-deal the 384 x 168 registers of the launch: with 168 the causal pairs spill 156 bytes (32 heads x 4096: 149 us, re-dealt
  // 138; 8 x 32768: 1960, 1845).  At d = 64 it does not pay (60.4 -> 62 us).
  static constexpr int kRegsSoftmax = 216, kRegsAux = 72;
  static_assert(2 * kRegsSoftmax + kRegsAux <= 3 * 168, "register shares");
  static constexpr int kPartF = D + 4;                 // row stride (floats) of a part in the cluster merge
  static_assert(256 * 4 * kPartF <= 2 * kTileBytes + kStages * 2 * kTileBytes, "the cluster merge goes over the Q and K / V tiles");
};

// TMEM columns of the scores and the probabilities.  At d = 64 there is room for S_0, S_1, P~_0 and P~_1.  At d = 128 there is
// not.  With P~_t over S_t a warpgroup's key tile is a serial chain of scores (512 clk), softmax (2600) and P~_t V (512), since the
// next scores have to wait for the last product: 3900 clk for two tiles in flight.  MODE 4, 5 and 6 keep P~_0 and P~_1 apart and
// one score tile that the warpgroups, half a tile apart, use in turn: it is free again as soon as one of them has copied its
// scores to registers, and the other's are computed while that one is in its exponentials.  Bound then by the exponentials of
// two warps per scheduler (2900 clk).  Measured (forward alone, calls back to back in a graph), P~ over S -> one score tile: pairs,
// causal: 8 heads x 32768: 2260 -> 1845 us; 32 x 4096: 167 -> 138; 96 x 1000: 49.0 -> 42.0; 256 x 500: 50.9 -> 43.6; not causal: 32 x
// 8192: 1050 -> 912; single tiles, causal: 8 x 4096: 42.6 -> 36; 8 x 2300: 25.3 -> 21.1; 24 packed documents, 16676 rows, 8 heads: 75.5
// -> 68.6; clusters and folded heads: 8 x (16, 4 heads) x 16 queries behind 8192 keys: 37.0 -> 29.9; 4 x 8 x 1 behind 16384: 58.1 ->
// 45.4; 2 x 1000 behind 20000: 64.8 -> 42.7; 16 x (32, 8) x 1 behind 1000: 17.8 -> 13.6; 64 x (32, 8) x 64 behind 2048: 262 -> 204.
// Where the second warpgroup would only wait for its first scores the old form is kept: tiles of one or two key tiles
// (64 heads x 384, causal: 12.3 -> 13.3; 200 documents of 30 to 300 rows, 16 heads: 218 -> 227; 1000 heads x 64: 35.5 -> 37.8),
// folded heads and clusters with fewer than four to a CTA (2 x (64, 8) x 100 behind 300: 9.4 -> 10.2).
template <int D, int MODE>
struct FwdTmem {
  static constexpr bool kSepP = (D == 64) || MODE == 4 || MODE == 5 || MODE == 6;   // P~ in its own columns
  static constexpr bool kSharedS = kSepP && D == 128;              // one score tile for both warpgroups
  static constexpr uint32_t kSStride = kSharedS ? 0 : 128;         // S_t at kSStride t
  static constexpr uint32_t kColP = !kSepP ? 0 : kSharedS ? 128 : 384, kPStride = kSepP ? 64 : 128;   // P~_t at kColP + kPStride t
};

enum FwdWaitCode {
  kFwdWaitQ = 0x11, kFwdWaitK = 0x12, kFwdWaitV = 0x13, kFwdWaitKVEmpty = 0x14, kFwdWaitS = 0x15, kFwdWaitP = 0x16,
  kFwdWaitPV = 0x17, kFwdWaitSFree = 0x18, kFwdWaitOFree = 0x19, kFwdWaitQFree = 0x1a, kFwdWaitMerge = 0x1c
};


// z = exp2(fl32[(x - x_max) (alpha log2 e)]) for the 128 columns of one row (two columns per packed FP32 instruction:
// the subtraction and the scale keep their separate roundings, add.rn / mul.rn; the fused variant of
// Eq. "historical-fma" is one fma.rn), BF16 pairs stored to TMEM at tP, returns the FP32 row sum of z (four packed
// partial sums).
template <bool FMA_SOFTMAX>
__device__ __forceinline__ float softmax_exp_store(const uint32_t (&xr)[4][32], uint32_t tP, float m_new, float scale_log2, float m_scaled) {
  const uint64_t negm2 = f32x2(-m_new, -m_new), scale2 = f32x2(scale_log2, scale_log2), negms2 = f32x2(-m_scaled, -m_scaled);
  uint64_t rs2[2] = {f32x2(0.f, 0.f), f32x2(0.f, 0.f)};
#pragma unroll
  for (int c = 0; c < 4; ++c) {
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

// MODE: 0 = pairs of query tiles (of heads with one tile), 2 = single tiles with the key range split between the warpgroups, 3 = single tiles with the key
// range split over the warpgroups of a cluster of CTAs (one tile per cluster; the parts of all CTAs are merged through
// distributed shared memory), 4 = as 2, 5 = as 0, 6 = as 3, with separate rings for K and V and the scores of both warpgroups in one
// place.  All at d = 128; at d = 64 only 3, everything else is attn_fwd_w64.cuh's.
template <int D, bool CAUSAL, bool FMA_SOFTMAX, int MODE>
__global__ void __launch_bounds__(384, 1)
attn_fwd_kernel(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmK,
                const __grid_constant__ CUtensorMap tmV, const __grid_constant__ CUtensorMap tmO,
                __nv_bfloat16 *__restrict__ Og, const int4 *__restrict__ plan, float *__restrict__ LSE, int N, int Nk, int BH, int Hq, int G, int fold_rows, int tiles_per_item, int total_items, const ItemOrder order, float scale_log2, float alpha,
                int *status) {
  // fold > 0 (cluster mode only): the query axis of a KV head is its G query heads' rows laid end to end, `fold` rows each
  // (grouped queries with few rows); row r then sees the keys of query r mod fold.
  using C = FwdCfg<D>;
  constexpr int S = C::kStages;
  constexpr bool kCluster = (MODE == 3 || MODE == 6);
  // Separate K and V rings: with one ring the next K waits for the whole softmax and P~V of its stage, which is what a ring of
  // two stages (d = 128) is bound by while the warpgroups work on two key tiles.  Measured, one ring -> two: 8 heads x 4096 x 128, causal:
  // 49.1 -> 41.4 us; 12 packed pairs (4000 queries, 9000 keys, 12 heads): 62.2 -> 51.5.  With few key tiles to an item (fwd_separate_rings
  // in host_rules.h), with more stages or where both stages hold one tile's work, the second commit per key tile and the
  // thread that polls both rings cost more than they give (200 packed documents of 30 to 300 rows, 16 heads, d = 128: 230 -> 270 us;
  // 16 heads x 4096 x 64: 60.5 -> 62.5; clusters at d = 64: 33.0 -> 38).  With the scores in one place they pay at every length of
  // pairs: 32 heads x 4096, causal: 159 -> 141; 32 x 2048: 72.5 -> 66.0.
  constexpr bool kSepRings = (MODE == 4 || MODE == 5 || MODE == 6);
  using M = FwdTmem<D, MODE>;
  constexpr bool kMoveRegs = M::kSharedS;
  const int fold = kCluster ? fold_rows : 0;
  extern __shared__ uint8_t smem_raw[];
  uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t *sQ = smem;                              // tile 0, then tile 1 (each later reused to stage O_t)
  uint8_t *sKV = sQ + 2 * C::kTileBytes;            // stage s: K tile, then V tile

  __shared__ int s_item[4][2];                     // rank and head of an item, from the Q loader to the softmax warps
  __shared__ uint64_t bar_q_full[2], bar_q_free[2], bar_k_full[S], bar_v_full[S], bar_k_empty[S], bar_v_empty[S];
  __shared__ uint64_t bar_s_full[2], bar_s_free[2], bar_p_ready[2], bar_pv_done[2], bar_o_free[2], bar_merge, bar_drain[2];
  __shared__ float s_m1[2][128], s_l1[2][128];   // split mode: running maximum and normaliser of the second warpgroup, by item parity (with a cluster: of both)
  __shared__ float s_pm[kCluster ? 256 : 1], s_pl[kCluster ? 256 : 1];   // cluster merge: every part's maximum and normaliser for this CTA's rows
  __shared__ uint32_t tmem_base_smem;
  __shared__ int cta_abort, cta_skip;

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) cta_skip = *reinterpret_cast<volatile int *>(status);
  __syncthreads();
  if (MODE == 5 && cta_skip != 0) { griddep_wait(); return; }   // see below

  const int n_qt = (N + C::kBlockM - 1) / C::kBlockM;   // the last tile may be ragged: rows past N load as zero, stores clip
  const int TPI = tiles_per_item;                  // 2: a pair of query tiles per work item; 1: single tiles, key range split
  constexpr bool split = (MODE != 0 && MODE != 5);              // one query tile; warpgroup t takes the key tiles j = t (mod 2), merged at the end
  // Key tile j of the item belongs to CTA (j / 2) mod ncta of the cluster (ncta = 1 without a cluster), warpgroup j mod 2.
  const int ncta = kCluster ? cluster_size() : 1, crank = kCluster ? cluster_rank() : 0;
  // The roles step through this CTA's key tiles alone.  (Walking over all of them with a division by ncta at each took an issuing
  // warp longer than its products.)
  const int j_first = 2 * crank;
  auto j_next = [&](int j) { return kCluster && (j & 1) ? j + 2 * ncta - 1 : j + 1; };
  const int n_pairs = (n_qt + TPI - 1) / TPI;
  AbortState ab{status, &cta_abort};
  if (threadIdx.x == 0) {
    cta_abort = kCluster ? cta_skip : 0;
    mbar_init(&bar_merge, 128);
    // Whenever a warp reads a slot (after an abort it may be too early or too late), it finds an item of this launch.
    for (auto &slot : s_item) slot[0] = slot[1] = 0;
    for (int b = 0; b < 2; ++b) {
      mbar_init(&bar_q_full[b], 1);
      mbar_init(&bar_q_free[b], 4 * tiles_per_item);    // one arrival per warp and query tile slot: its O store has left shared memory
    }
    for (int s = 0; s < S; ++s) { mbar_init(&bar_k_full[s], 1); mbar_init(&bar_v_full[s], 1); mbar_init(&bar_k_empty[s], 1); mbar_init(&bar_v_empty[s], 1); }
    for (int t = 0; t < 2; ++t) {
      mbar_init(&bar_drain[t], 1);
      mbar_init(&bar_s_full[t], 1); mbar_init(&bar_s_free[t], 128); mbar_init(&bar_p_ready[t], 128); mbar_init(&bar_pv_done[t], 1); mbar_init(&bar_o_free[t], 128);
    }
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
  // An earlier wait gave up: drain the rest of the grid quickly, but not past the kernel before this one, for whose end the
  // next kernel in the stream relies on this one.  The CTAs of a cluster wait for one another at the end, so they run on with
  // every wait falling through instead.  Where this return stands changes the code of the softmax loop.  Above, behind a
  // griddep_wait of its own, calls of one or two key tiles per item are up to 3 % slower (64 x 16 heads x 100 x 64: 31.7 -> 32.8 us); here,
  // pairs with separate rings are no faster (8 heads x 32768 x 128, causal: 1846 and 1850 us).
  if (!kCluster && MODE != 5 && cta_skip != 0) {
    __syncthreads();
    if (warp == 1) tmem_dealloc(tmem_base, C::kTmemCols);
    return;
  }

  // Work items ordered by decreasing work (causal: last pair first).  Item -> (sequence, first query tile, tiles) and head.
  // Dense calls: one sequence [0, N) per head, items are pairs (or single tiles); packed calls: single tiles from the plan.
  // qt0: index of the first query tile inside its sequence; nq: query tiles; n_kt: key tiles walked; kseq0, klen: the keys.
  // Causal support of query i: keys j <= i + off with off = klen - len (the diagonal ends at the last query and last key).
  struct Item { int seq0, len, qt0, nq, n_kt, kseq0, klen, off; };
  auto tix = [&](int lin) { return order.rank(lin); };
  auto hix = [&](int lin) { return order.head(lin); };
  TileSched sched(total_items, order.solo, ncta);
  auto decode_rank = [&](int rank) {       // rank: position of the item's tile (pair) in its head's list, longest first
    Item it;
    if (plan != nullptr) {
      const TileInfo ti = tile_info(plan, rank, 0, N, Nk);
      it.seq0 = ti.seq0; it.len = ti.seq_end - ti.seq0; it.qt0 = (ti.row0 - ti.seq0) / C::kBlockM; it.nq = 1;
      it.kseq0 = ti.oseq0; it.klen = ti.oseq_end - ti.oseq0;
    } else {
      const int pair = CAUSAL ? (n_pairs - 1 - rank) : rank;
      it.seq0 = 0; it.len = N; it.qt0 = TPI * pair; it.nq = min(TPI, n_qt - it.qt0);
      it.kseq0 = 0; it.klen = Nk;
    }
    it.off = it.klen - (fold > 0 ? fold : it.len);
    // key tiles up to the last key the item's last row sees; at least one (fully masked if the item sees no key at all)
    const int kend = (CAUSAL && fold == 0) ? min(it.klen, (it.qt0 + it.nq) * C::kBlockM + it.off) : it.klen;
    it.n_kt = max(1, (max(kend, 0) + C::kBlockN - 1) / C::kBlockN);
    return it;
  };
  auto decode = [&](int lin) { return decode_rank(tix(lin)); };
  // query tile t of the item takes part in key step j?  (key tile 0 always, so that every tile has a first step)
  auto active = [&](const Item &it, int t, int j) {
    return t < it.nq && (!CAUSAL || fold > 0 || j <= max(0, ((it.qt0 + t) * C::kBlockM + C::kBlockM - 1 + it.off) >> 7));
  };

  // Cluster mode, a tile of at most 64 (32) rows: the second warpgroup's copy of the tile sits 64 (32) lanes further up, so
  // that the live warps of the two warpgroups are on different schedulers.
  auto lane_shift = [&](const Item &it, int t) {
    const int rows = it.len - it.qt0 * C::kBlockM;
    return kCluster && t == 1 && rows <= 64 ? (rows <= 32 ? 32 : 64) : 0;
  };

  // Q buffers: a pair item fills both tile slots of the one buffer; single-tile items (split mode) alternate between the
  // two slots, so that the next item's Q is loaded, and its first scores are computed, during this item's epilogue.
  auto q_buf = [&](int ti) { return split ? (ti & 1) : 0; };
  auto q_use = [&](int ti) { return split ? (ti >> 1) : ti; };      // how often the buffer has been used before item ti

  if (warp < 4) {
  if constexpr (kMoveRegs) setmaxnreg_dec<C::kRegsAux>();
  if (warp == 0) {
    // ---------------------------------------------------------------- TMA producer of K_j, V_j
    // With separate rings a K tile is free as soon as its scores are complete, a V tile only when the probabilities of its
    // key tile have been multiplied, a whole softmax later.  One thread feeds both rings and takes whichever has a free
    // slot, so the next K is on its way while a V slot is still busy.
    if (kSepRings && lane == 0) {
      struct Cursor {
        TileSched sched;
        Item it;
        int j, kvh, g;
        bool more;
      };
      auto next_item = [&](Cursor &c) {
        const int lin = c.sched.next();
        c.more = lin >= 0;
        if (!c.more) return;
        c.it = decode(lin);
        c.kvh = kv_head_of(hix(lin), Hq, G);                 // grouped-query: the group's shared K / V head
        c.j = j_first;
      };
      auto settle = [&](Cursor &c) {                         // on to the next key tile of this CTA's
        while (c.more && c.j >= c.it.n_kt) next_item(c);
      };
      auto feed = [&](Cursor &c, uint64_t *full, uint64_t *empty, const CUtensorMap *map, uint8_t *ring) {
        const int st = c.g % S;
        if (!c.more || (c.g >= S && !mbar_test_wait(&empty[st], ((c.g / S) - 1) & 1))) return false;
        mbar_expect_tx(&full[st], C::kTileBytes);
        for (int s = 0; s < C::kSlabs; ++s)
          tma_load_3d(ring + st * 2 * C::kTileBytes + s * C::kSlabBytes, map, &full[st], s * 64, c.it.kseq0 + c.j * C::kBlockN, c.kvh);
        ++c.g;
        c.j = j_next(c.j);
        settle(c);
        return true;
      };
      Cursor ck{sched, Item{}, 0, 0, 0, true}, cv = ck;
      next_item(ck); settle(ck);
      cv = ck;
      BoundedIdle idle;
      while (ck.more || cv.more) {
        const bool fed_k = feed(ck, bar_k_full, bar_k_empty, &tmK, sKV);
        const bool fed_v = feed(cv, bar_v_full, bar_v_empty, &tmV, sKV + C::kTileBytes);
        if (!idle.go_on(fed_k || fed_v, ab, kFwdWaitKVEmpty)) break;
      }
      // Every load is consumed by an MMA the epilogue waits for, so nothing is in flight at exit unless the
      // CTA aborted; then give the copies a bounded chance to land before shared memory is released.
      if (cta_abort) {
        for (int q = (ck.g > S ? ck.g - S : 0); q < ck.g; ++q)
          for (int spin = 0; spin < 100000 && !mbar_try_wait(&bar_k_full[q % S], (q / S) & 1); ++spin) {}
        for (int q = (cv.g > S ? cv.g - S : 0); q < cv.g; ++q)
          for (int spin = 0; spin < 100000 && !mbar_try_wait(&bar_v_full[q % S], (q / S) & 1); ++spin) {}
      }
    }
    if (!kSepRings && lane == 0) {
      int g = 0;
      for (int lin = sched.next(); lin >= 0; lin = sched.next()) {
        const Item it = decode(lin);
        const int bh = hix(lin), T = it.n_kt;
        for (int j = j_first; j < T; j = j_next(j)) {
          const int st = g % S;
          if (g >= S) mbar_wait(&bar_v_empty[st], ((g / S) - 1) & 1, ab, kFwdWaitKVEmpty);
          uint8_t *dK = sKV + st * 2 * C::kTileBytes, *dV = dK + C::kTileBytes;
          const int kvh = kv_head_of(bh, Hq, G), krow = it.kseq0 + j * C::kBlockN;   // grouped-query: the group's shared K / V head
          mbar_expect_tx(&bar_k_full[st], C::kTileBytes);
          for (int s = 0; s < C::kSlabs; ++s) tma_load_3d(dK + s * C::kSlabBytes, &tmK, &bar_k_full[st], s * 64, krow, kvh);
          mbar_expect_tx(&bar_v_full[st], C::kTileBytes);
          for (int s = 0; s < C::kSlabs; ++s) tma_load_3d(dV + s * C::kSlabBytes, &tmV, &bar_v_full[st], s * 64, krow, kvh);
          ++g;
        }
      }
      if (cta_abort) {
        for (int q = (g > S ? g - S : 0); q < g; ++q) {
          for (int spin = 0; spin < 100000 && !mbar_try_wait(&bar_k_full[q % S], (q / S) & 1); ++spin) {}
          for (int spin = 0; spin < 100000 && !mbar_try_wait(&bar_v_full[q % S], (q / S) & 1); ++spin) {}
        }
      }
    }
  } else if (warp == 3) {
    // ---------------------------------------------------------------- TMA loader of the stationary Q pair
    if (lane == 0) {
      int ti = 0;
      for (int lin = sched.next(); lin >= 0; lin = sched.next(), ++ti) {
        const Item it = decode(lin);
        const int bh = hix(lin), tiles = it.nq;
        const int qb = q_buf(ti), use = q_use(ti);
        if (use >= 1) mbar_wait(&bar_q_free[qb], (use - 1) & 1, ab, kFwdWaitQFree, tile_wait_budget(2LL * (Nk / C::kBlockN + 1)));   // up to two tiles
        // The softmax warps (168 registers, the kernel's tightest code) take the item's rank and head from here instead
        // of decoding the item number themselves; the barrier's completion publishes the two words.  The loader is at
        // most two items ahead of them, the ring has four entries.
        s_item[ti & 3][0] = tix(lin);
        s_item[ti & 3][1] = bh;
        const int copies = lane_shift(it, 1) > 0 ? 2 : tiles;   // shifted: the same tile once more
        mbar_expect_tx(&bar_q_full[qb], copies * C::kTileBytes);
        for (int t = 0; t < copies; ++t)
          for (int s = 0; s < C::kSlabs; ++s)
            tma_load_3d(sQ + (qb + t) * C::kTileBytes + s * C::kSlabBytes, &tmQ, &bar_q_full[qb], s * 64,
                        it.seq0 + (kCluster ? it.qt0 * C::kBlockM - lane_shift(it, t) : (it.qt0 + t) * C::kBlockM), bh);
      }
      if (cta_abort)
        for (int q = (ti > 2 ? ti - 2 : 0); q < ti; ++q)
          for (int spin = 0; spin < 100000 && !mbar_try_wait(&bar_q_full[q_buf(q)], q_use(q) & 1); ++spin) {}
    }
  } else if (warp == 1) {
    // ---------------------------------------------------------------- tensor-core issuer 1: S_t = Q_t K_j^T
    // The whole warp runs this loop so that every address stays provably warp-uniform (descriptor operands
    // then live in uniform registers); one elected lane issues the MMAs and commits.
    constexpr uint32_t idesc_s = idesc_bf16_f32(128, 128, 0, 0);   // both operands K-major
    const SmemDesc dscQ0 = make_smem_desc(smem_u32(sQ), 16, 1024);
    const SmemDesc dscK0 = make_smem_desc(smem_u32(sKV), 16, 1024);
    int g = 0, ti = 0, cnt[2] = {0, 0}, last = -1;
    for (int lin = sched.next(); lin >= 0; lin = sched.next(), ++ti) {
      const Item it = decode(lin);
      const int T = it.n_kt;
      const int qb = q_buf(ti);
      mbar_wait(&bar_q_full[qb], q_use(ti) & 1, ab, kFwdWaitQ);
      for (int j = j_first; j < T; j = j_next(j)) {
        const int st = g % S;
        mbar_wait(&bar_k_full[st], (g / S) & 1, ab, kFwdWaitK);
        const SmemDesc dscK = dscK0.advanced(st * 2 * C::kTileBytes);
#pragma unroll
        for (int t = 0; t < 2; ++t) {
          if (split ? ((j & 1) != t) : !active(it, t, j)) continue;
          // S_t may be overwritten once its previous contents are dead: copied to registers by the softmax (P~ has its
          // own columns), or, when P~ lives in the same columns, consumed by the previous P~V product.
          // With one score tile for both warpgroups those are the scores issued last, whoever's they are.
          if (M::kSharedS) {
            if (last >= 0) mbar_wait(&bar_s_free[last], (cnt[last] - 1) & 1, ab, kFwdWaitSFree);
            last = t;
          } else if (cnt[t] > 0) {
            if (M::kSepP) mbar_wait(&bar_s_free[t], (cnt[t] - 1) & 1, ab, kFwdWaitSFree);
            else          mbar_wait(&bar_pv_done[t], (cnt[t] - 1) & 1, ab, kFwdWaitSFree);
          }
          tc_fence_after();
          const SmemDesc dscQ = dscQ0.advanced((split ? (lane_shift(it, t) > 0 ? t : qb) : t) * C::kTileBytes);
          if (elect_one_sync()) {
#pragma unroll
            for (int k = 0; k < D / 16; ++k) {
              const uint32_t off = (k / 4) * C::kSlabBytes + (k % 4) * 32;
              umma_ss(tmem_base + C::kColS + M::kSStride * t, dscQ.at(off), dscK.at(off), idesc_s, k > 0);
            }
            umma_commit(&bar_s_full[t]);
          }
          __syncwarp();
          ++cnt[t];
        }
        if (kSepRings) {
          if (elect_one_sync()) umma_commit(&bar_k_empty[st]);   // every score product that reads this K tile has been issued
          __syncwarp();
        }
        ++g;
      }
    }
    drain_mmas_if_aborted(&bar_drain[0], ab);
  } else if (warp == 2) {
    // ---------------------------------------------------------------- tensor-core issuer 2: O_t += P~_t V_j
    constexpr uint32_t idesc_o = idesc_bf16_f32(128, D, 0, 1);     // V is MN-major (d contiguous)
    const SmemDesc dscV0 = make_smem_desc(smem_u32(sKV + C::kTileBytes), C::kSlabBytes, 1024);
    int g = 0, ti = 0, cnt[2] = {0, 0};
    for (int lin = sched.next(); lin >= 0; lin = sched.next(), ++ti) {
      const Item it = decode(lin);
      const int T = it.n_kt;
      for (int j = j_first; j < T; j = j_next(j)) {
        const int st = g % S;
        mbar_wait(&bar_v_full[st], (g / S) & 1, ab, kFwdWaitV);
        const SmemDesc dscV = dscV0.advanced(st * 2 * C::kTileBytes);
#pragma unroll
        for (int t = 0; t < 2; ++t) {
          if (split ? ((j & 1) != t) : !active(it, t, j)) continue;
          const bool first = split ? (j < 2 * crank + 2) : (j == 0);     // first product into O_t in this work item
          if (first && ti > 0) mbar_wait(&bar_o_free[t], (ti - 1) & 1, ab, kFwdWaitOFree);   // previous epilogue has read O_t
          mbar_wait(&bar_p_ready[t], cnt[t] & 1, ab, kFwdWaitP);
          tc_fence_after();
          const uint32_t tP = tmem_base + M::kColP + M::kPStride * t;
          const uint32_t acc = first ? 0u : 1u;
          if (elect_one_sync()) {
#pragma unroll
            for (int k = 0; k < C::kBlockN / 16; ++k)
              umma_ts(tmem_base + C::kColO + D * t, tP + 8 * k, dscV.at(k * 2048), idesc_o, k > 0 ? 1u : acc);
            umma_commit(&bar_pv_done[t]);
          }
          __syncwarp();
          ++cnt[t];
        }
        if (elect_one_sync()) umma_commit(&bar_v_empty[st]);     // every product that reads this V tile has been issued
        __syncwarp();
        ++g;
      }
    }
    drain_mmas_if_aborted(&bar_drain[1], ab);
  }
  } else {
    if constexpr (kMoveRegs) setmaxnreg_inc<C::kRegsSoftmax>();
    // ---------------------------------------------------------------- softmax: warpgroup t <-> query tile t, thread <-> row
    const int t = (warp - 4) >> 2;
    const int row = 32 * (warp & 3) + lane;
    const uint32_t lane_addr = static_cast<uint32_t>(32 * (warp & 3)) << 16;
    const uint32_t tS = tmem_base + C::kColS + M::kSStride * t + lane_addr;
    const uint32_t tO = tmem_base + C::kColO + D * t + lane_addr;
    const uint32_t tP = tmem_base + M::kColP + M::kPStride * t + lane_addr;
    int ti = 0, cnt = 0;
    for (int lin = sched.next(); lin >= 0; lin = sched.next(), ++ti) {
      const int qb = q_buf(ti);
      mbar_wait(&bar_q_full[qb], q_use(ti) & 1, ab, kFwdWaitQ);   // the item's Q has landed, and with it its description
      const Item it = decode_rank(s_item[ti & 3][0]);
      const int bh = s_item[ti & 3][1], T = it.n_kt;
      const int qt = it.qt0 + (split ? 0 : t);        // this warpgroup's query tile inside the sequence
      // Masking, reduced to two numbers per tile: column c of key tile j is outside the row's support when
      // 128 j + c > rk, with rk the last key the row sees (causal diagonal and end of the keys, whichever comes first);
      // no key tile before jm needs the test for any row of the tile.
      const int trow = row - lane_shift(it, t);       // row inside the tile
      const int q_lo = fold > 0 ? 0 : qt * C::kBlockM, q_row = fold > 0 ? (qt * C::kBlockM + trow) % fold : qt * C::kBlockM + trow;   // first query of the tile, this row's query
      const int rk = CAUSAL ? min(q_row + it.off, it.klen - 1) : it.klen - 1;
      const int jl = (CAUSAL && fold == 0) ? max(0, (qt * C::kBlockM + C::kBlockM - 1 + it.off) >> 7) : T;   // last key tile of this query tile
      const int jm = CAUSAL ? min((q_lo + it.off + 1) >> 7, it.klen >> 7) : (it.klen >> 7);
      // A warp none of whose rows exist (a short block of queries) only keeps the barriers going.
      const bool live = trow >= 0 && qt * C::kBlockM + trow - lane < it.len;
      if (!split && t >= it.nq) {
        // Odd number of query tiles: the last pair has no second tile.  This warpgroup is in step with the item (it has
        // waited for its Q above), so it may hand back the slot without any barrier running ahead of its waiters.
        if (lane == 0) mbar_arrive(&bar_q_free[0]);
        mbar_arrive(&bar_o_free[t]);
        continue;
      }
      float m_run = -INFINITY, l_run = 0.f;
#ifdef GPROJ_TRACE
      const unsigned long long ev_n0 = global_ns(); const long long ev_c0 = clock64();
#endif
      const int cnt_item0 = cnt;
      for (int j = split ? 2 * crank + t : 0; j < T; j += split ? 2 * ncta : 1) {
        const bool first = split ? (j < 2 * crank + 2) : (j == 0);     // this warpgroup's first key tile of the item
        if (!split && j > jl) continue;               // causal: the first tile of the pair ends one key tile earlier
        mbar_wait(&bar_s_full[t], cnt & 1, ab, kFwdWaitS);
        tc_fence_after();
        if (kCluster && !live) {
          if (M::kSepP) mbar_arrive(&bar_s_free[t]);
          if (!first) mbar_wait(&bar_pv_done[t], (cnt - 1) & 1, ab, kFwdWaitPV);
          mbar_arrive(&bar_p_ready[t]);
          ++cnt;
          continue;
        }
        uint32_t xr[4][32];
#pragma unroll
        for (int c = 0; c < 4; ++c) tmem_ld32(tS + 32 * c, xr[c]);
        tmem_wait_ld();
        if (M::kSepP) { tc_fence_before(); mbar_arrive(&bar_s_free[t]); }   // the next S_t may be issued while this one is in the ALUs
        // Keys beyond the causal diagonal, and the zero-filled columns past the last key of a ragged tile, get -inf.
        if (j >= jm) {
          const int lim = rk - j * C::kBlockN;
#pragma unroll
          for (int c = 0; c < 4; ++c)
#pragma unroll
            for (int i = 0; i < 32; ++i)
              if (32 * c + i > lim) xr[c][i] = 0xff800000u;
        }
        // Row maximum over eight independent chains of three-input maxima (only two softmax warps share a scheduler, so a
        // 128-long dependent chain would be pure latency).
        float mxp[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) mxp[i] = fmaxf(__uint_as_float(xr[0][i]), __uint_as_float(xr[0][8 + i]));
#pragma unroll
        for (int e = 16; e < 128; e += 16)
#pragma unroll
          for (int i = 0; i < 8; ++i)
            mxp[i] = fmax3(mxp[i], __uint_as_float(xr[(e + i) >> 5][(e + i) & 31]), __uint_as_float(xr[(e + 8 + i) >> 5][(e + 8 + i) & 31]));
        // The floor keeps the maximum finite for a row that has seen no key yet (unequal lengths: rows before the causal
        // diagonal reaches key 0), so that such a row gives z = exp2(-inf) = 0 instead of NaN from (-inf) - (-inf).
        const float mx = fmax3(fmax3(mxp[0], mxp[1], mxp[2]), fmax3(mxp[3], mxp[4], mxp[5]), fmax3(mxp[6], mxp[7], kFwdMaxFloor));
        // Lazy maximum: the running maximum is only raised when the tile's maximum exceeds it by more than 8 in the
        // base-two exponent domain; otherwise the stale value stays (z <= 2^8, harmless in FP32 / BF16: O = acc / l and
        // LSE = alpha m + ln l do not depend on which reference m was subtracted) and neither l nor the accumulator
        // needs a rescale.  The first tile always sets it (m_run = -inf).  The fused variant always takes the true
        // running maximum, so that it is the arithmetic of Eq. "historical-fma" and nothing else.
        float m_new = fmaxf(m_run, mx);
#ifndef GPROJ_FWD_EAGER_MAX
        if (!FMA_SOFTMAX && __fmul_rn(__fsub_rn(m_new, m_run), scale_log2) <= 8.0f) m_new = m_run;
#endif
        const float corr = fast_exp2(__fmul_rn(__fsub_rn(m_run, m_new), scale_log2));
        // FMA_SOFTMAX reproduces the native fused form of Eq. "historical-fma": z = exp2(fma(x, a, -fl32(x_max a))),
        // in which x a is not rounded separately, so the largest score need not map to exactly zero.
        const float m_scaled = __fmul_rn(m_new, scale_log2);
        // P~ of the previous key tile must have been consumed (and O_t updated) before either is touched
        if (!first) { mbar_wait(&bar_pv_done[t], (cnt - 1) & 1, ab, kFwdWaitPV); tc_fence_after(); }
        const float rs = softmax_exp_store<FMA_SOFTMAX>(xr, tP, m_new, scale_log2, m_scaled);
        l_run = l_run * corr + rs;
        if (!first && __any_sync(0xffffffffu, m_new != m_run)) {
#pragma unroll
          for (int c = 0; c < D / 32; ++c) {
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
        mbar_arrive(&bar_p_ready[t]);
        ++cnt;
      }
#ifdef GPROJ_TRACE
      const unsigned long long ev_n2 = global_ns();
#endif
      // ---- epilogue: O = BF16(acc / l) staged in the TMA layout over this tile's Q, LSE = alpha x_max + ln l
      if (cnt > cnt_item0) { mbar_wait(&bar_pv_done[t], (cnt - 1) & 1, ab, kFwdWaitPV); tc_fence_after(); }
      if (kCluster) {
        // the merge is below, by all threads of the cluster
        if (live) {
          s_m1[t][trow] = m_run;
          s_l1[t][trow] = l_run;
        }
        named_bar_sync(3, 256);                    // both warpgroups' products are complete: Q, K and V are consumed
        if (live) {
          float *part = reinterpret_cast<float *>(smem) + (t * 128 + trow) * C::kPartF;
#pragma unroll
          for (int c = 0; c < D / 16; ++c) {
            uint32_t o[16];
            tmem_ld16(tO + 16 * c, o);
            tmem_wait_ld();
            const bool has = l_run != 0.f;         // otherwise the accumulator may never have been written; a NaN goes on to the output
#pragma unroll
            for (int v = 0; v < 4; ++v)
              *reinterpret_cast<uint4 *>(part + 16 * c + 4 * v) = has ? make_uint4(o[4 * v], o[4 * v + 1], o[4 * v + 2], o[4 * v + 3]) : make_uint4(0u, 0u, 0u, 0u);
          }
        }
        tc_fence_before();
        break;
      }
      if (split && t == 1) {
        // hand this half's statistics to warpgroup 0, which merges the two accumulators (l = 0: no key tiles here).
        // With two Q slots this warpgroup could finish a second item before warpgroup 0 has looked at the first one's
        // hand-over, and the merge barrier would be two phases ahead of its waiter; so it first waits until
        // warpgroup 0 has read the previous item's accumulators.
        if (ti > 0) mbar_wait(&bar_o_free[1], (ti - 1) & 1, ab, kFwdWaitOFree);
        s_m1[ti & 1][row] = m_run;
        s_l1[ti & 1][row] = l_run;
        tc_fence_before();
        mbar_arrive(&bar_merge);
#ifdef GPROJ_TRACE
        if (row == 0) tile_event(21, lin, T, ev_n0, ev_n0, ev_n2, global_ns(), ev_c0, clock64());
#endif
        continue;
      }
      // Split mode: O = (O_0 s_0 + O_1 s_1) / (l_0 s_0 + l_1 s_1) with s_t = exp2((m_t - max(m_0, m_1)) alpha log2 e).
      const bool has1 = split && T >= 2;               // the second warpgroup had at least one key tile
      float a0 = (l_run > 0.f) ? 1.0f / l_run : 0.f, a1 = 0.f;   // a row with an empty support has l = 0: O = 0
      if (split) {
        mbar_wait(&bar_merge, ti & 1, ab, kFwdWaitMerge);
        tc_fence_after();
        if (has1) {
          const float m1 = s_m1[ti & 1][row], l1 = s_l1[ti & 1][row];
          const float m = fmaxf(m_run, m1);
          const float s0 = fast_exp2(__fmul_rn(__fsub_rn(m_run, m), scale_log2)), s1 = fast_exp2(__fmul_rn(__fsub_rn(m1, m), scale_log2));
          l_run = fmaf(l_run, s0, l1 * s1);
          m_run = m;
          const float inv = (l_run > 0.f) ? 1.0f / l_run : 0.f;   // neither half has seen a key: O = 0
          a0 = s0 * inv;
          a1 = s1 * inv;
        }
      }
      const float inv_l = has1 ? 1.0f : a0;            // with two halves the weights a_0, a_1 already carry 1 / l
      uint8_t *stage = sQ + (split ? qb : t) * C::kTileBytes;   // no MMA reads this Q tile any more
#pragma unroll
      for (int c = 0; c < D / 32; ++c) {
        uint32_t o[32];
        tmem_ld32(tO + 32 * c, o);
        if (has1) {
          uint32_t o1[32];
          tmem_ld32(tO + D + 32 * c, o1);              // O_1 sits D columns after O_0, same lanes
          tmem_wait_ld();
#pragma unroll
          for (int i = 0; i < 32; ++i) o[i] = __float_as_uint(fmaf(__uint_as_float(o1[i]), a1, __uint_as_float(o[i]) * a0));
        }
        tmem_wait_ld();
        const uint32_t slab = (c >> 1) * C::kSlabBytes;
#pragma unroll
        for (int v = 0; v < 4; ++v) {
          uint32_t pk[4];
#pragma unroll
          for (int w = 0; w < 4; ++w)
            pk[w] = pack_bf16x2(__uint_as_float(o[8 * v + 2 * w]) * inv_l, __uint_as_float(o[8 * v + 2 * w + 1]) * inv_l);
          *reinterpret_cast<uint4 *>(stage + slab + swz128_offset(row, 4 * (c & 1) + v)) = make_uint4(pk[0], pk[1], pk[2], pk[3]);
        }
      }
      tc_fence_before();
      mbar_arrive(&bar_o_free[t]);                     // O_t may be overwritten by the next work item
      if (split) mbar_arrive(&bar_o_free[1]);          // warpgroup 0 has read both accumulators
      const int qrow0 = it.seq0 + qt * C::kBlockM;      // first row of the tile inside the head
      if (qt * C::kBlockM + row < it.len) LSE[static_cast<size_t>(bh) * N + qrow0 + row] = (l_run > 0.f) ? fmaf(m_run, alpha, logf(l_run)) : INFINITY;
      // Every warp writes its own 32 rows out: after an abort the warps of a warpgroup may be at different items, and a barrier among
      // them, which has no limit, could wait for ever.
      const TileInfo tinfo{qrow0, it.seq0, it.seq0 + it.len, 0};
      if (tile_store_by_tma(tinfo, N)) {
        fence_proxy_async_smem();
        __syncwarp();
        if (lane == 0 && qt * C::kBlockM + row < it.len) {
          for (int sl = 0; sl < C::kSlabs; ++sl) tma_store_3d(&tmO, stage + sl * C::kSlabBytes + row * 128, sl * 64, qrow0 + row, bh);
          bulk_commit_group();
          bulk_wait_group_read0();
        }
      } else {
        // ragged last tile of a packed sequence that another sequence follows: rows past its end are not ours to write
        store_rows_clipped<D>(stage, C::kSlabBytes, Og + (static_cast<size_t>(bh) * N + qrow0) * D, row, it.len - qt * C::kBlockM);
        __syncwarp();
      }
      if (lane == 0) mbar_arrive(&bar_q_free[qb]);     // this tile's slot of the Q buffer may be reloaded
#ifdef GPROJ_TRACE
      if (row == 0) tile_event(20 + t, lin, T, ev_n0, ev_n0, ev_n2, global_ns(), ev_c0, clock64());
#endif
    }
  }

  if (kCluster) {
    // Merge of the 2 ncta partial results of the cluster's tile: O = sum_w O_w s_w / L with s_w = exp2((m_w - M) alpha log2 e),
    // M = max m_w, L = sum l_w s_w.  Every CTA has left its two parts in its own shared memory and finishes 128 / ncta of the
    // rows, reading the others' parts by whole rows, in a fixed order.  (Scaling the parts first and sending them row by
    // row, thread by thread, took 7 us from the last product to the result, 12 us at d = 128.  Measured with the lane shift, that ->
    // this: 8 x (16 query, 4 KV heads) x 16 queries behind 8192 keys, d = 64: 30.3 -> 27.2 us; d = 128: 43.4 -> 38.9; 16 x (32,
    // 8 heads) x 1 query behind 1000 keys, d = 64: 15.5 -> 13.0.)
    const int own = 128 / ncta, nsrc = 2 * ncta;
    cluster_sync();
    const Item it = decode(sched.c);
    const int bh = hix(sched.c), row0 = it.qt0 * C::kBlockM + crank * own;     // first of this CTA's rows
    if (threadIdx.x < 256) {
      const int w = threadIdx.x / own, r = crank * own + threadIdx.x % own;
      s_pm[threadIdx.x] = cluster_load_f32(cluster_map_shared(smem_u32(&s_m1[w & 1][r]), w >> 1));
      s_pl[threadIdx.x] = cluster_load_f32(cluster_map_shared(smem_u32(&s_l1[w & 1][r]), w >> 1));
    }
    __syncthreads();
    for (int i = threadIdx.x; i < own * (D / 4); i += C::kThreads) {
      const int r = i / (D / 4), c4 = i % (D / 4), qrel = row0 + r;
      if (qrel >= it.len) continue;
      const uint32_t src = smem_u32(smem) + static_cast<uint32_t>(((crank * own + r) * C::kPartF + 4 * c4) * 4);
      float M = kFwdMaxFloor;                                                   // a part without key tiles has m = -inf, l = 0
      for (int w = 0; w < nsrc; ++w) M = fmaxf(M, s_pm[w * own + r]);
      float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
      float L = 0.f;
#pragma unroll 4
      for (int c = 0; c < ncta; ++c) {                       // the two parts of CTA c
        const uint32_t from = cluster_map_shared(src, c);
        float v0[4], v1[4];
        cluster_load_f4(from, v0);
        cluster_load_f4(from + 128 * C::kPartF * 4, v1);
        const float e0 = fast_exp2(__fmul_rn(__fsub_rn(s_pm[2 * c * own + r], M), scale_log2)), e1 = fast_exp2(__fmul_rn(__fsub_rn(s_pm[(2 * c + 1) * own + r], M), scale_log2));
        L += s_pl[2 * c * own + r] * e0 + s_pl[(2 * c + 1) * own + r] * e1;
        acc.x = fmaf(v1[0], e1, fmaf(v0[0], e0, acc.x)); acc.y = fmaf(v1[1], e1, fmaf(v0[1], e0, acc.y));
        acc.z = fmaf(v1[2], e1, fmaf(v0[2], e0, acc.z)); acc.w = fmaf(v1[3], e1, fmaf(v0[3], e0, acc.w));
      }
      const float inv = L > 0.f ? 1.0f / L : 0.f;            // a row with an empty support: O = 0
      const size_t grow = static_cast<size_t>(bh) * N + it.seq0 + qrel;
      *reinterpret_cast<uint2 *>(Og + grow * D + 4 * c4) = make_uint2(pack_bf16x2(acc.x * inv, acc.y * inv), pack_bf16x2(acc.z * inv, acc.w * inv));
      if (c4 == 0) LSE[grow] = (L > 0.f) ? fmaf(M, alpha, logf(L)) : INFINITY;
    }
    cluster_sync();                                          // no CTA leaves while another one may still read its parts
  }

  tc_fence_before();
  __syncthreads();
  if (warp == 1) tmem_dealloc(tmem_base, C::kTmemCols);
}

}  // namespace gproj
