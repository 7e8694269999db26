// Rules by which the host chooses between kernels and launch shapes.  Plain C++, so that they can be checked without a GPU.
#pragma once

#include <algorithm>
#include <vector>

namespace gproj {

// The count that `query` writes, or none where it fails: a launch shape that the device cannot vouch for is not used, and the
// calls that do not need it run all the same.
template <typename Query>
int count_or_none(Query query) {
  int n = 0;
  return query(&n) ? std::max(n, 0) : 0;
}

// Key tiles that the query tiles of one sequence walk: all of them, or those up to the diagonal that ends at the last query and
// key; one where a tile sees no key.
inline long long fwd_key_tiles(int lq, int lk, bool causal) {
  const long long tq = (lq + 127LL) / 128, tk = std::max<long long>(1, (lk + 127LL) / 128);
  if (!causal || tq == 0) return tq * tk;
  const long long off = static_cast<long long>(lk) - lq, e = off >= 0 ? (off + 127) / 128 : -(-off / 128);   // off / 128, rounded up
  const long long ones = std::max<long long>(0, std::min(tq, -e));      // tiles before the diagonal reaches key 0, beside the next
  const long long n = tq - ones;                                        // the others: ones + 1 + e, ones + 2 + e, ... tq + e
  return ones + n * (ones + 1 + e + tq + e) / 2 - (n > 0 ? std::max<long long>(0, tq + e - tk) : 0);
}

// What an item of the forward costs beside its key tiles, in key tiles; for a pair of query tiles in ranks, of two key tiles each.
// Measured, in microseconds per item and per key tile: d = 64: 1.4 and 0.77; d = 128, single tiles: 3.1 and 1.45.  Pairs take 3 and 2.05,
// which would be 0.7; the 1.45 of an older kernel stays.  It groups ranks (tile_group_of) in 30 of 557 sizes where 0.7 does not: 88 heads x
// 3968 x 128, causal: 349 us (0.7: 352) in a short burst, 438 (391) under the power limit; 64 x 7424: 747 (790), 894 (874).  For the CTAs
// with one item (solo_ctas) 1.2 to 2.4 are alike.
inline double fwd_item_cost(int d, bool pairs) { return d == 64 ? 1.8 : pairs ? 1.45 : 2.1; }

// Forward at d = 128 with the key range of a tile split between the warpgroups: separate rings for K and V (see attn_fwd.cuh)?
// From three key tiles per item on (key_tiles, tiles: of one head, or of the items of one CTA; with one item per CTA: of the longest item).
// Measured, one ring -> two, 16 query / 4 KV heads, 40000 rows in sequences of one length, causal: 512 rows (2.5 key tiles per item)
// 228 -> 239 us, 640 (3.0) 256 -> 256, 1024 (4.5) 332 -> 312; not causal: 256 (2) 177 -> 190, 384 (3) 240 -> 234.  With the scores of both
// warpgroups in one place as well (FwdTmem): 64 heads x 384, causal (2.0) 12.3 -> 13.3, x 500 (2.5) 16.0 -> 15.6, not causal: 256 (2) 8.5
// -> 8.6, 384 (3) 17.5 -> 15.2; one item per CTA, causal: 16 x 500 (4) 10.6 -> 9.3, 16 x 300 (3) 8.7 -> 8.2, 16 x 200 (2) 7.0 -> 7.2.
inline bool fwd_separate_rings(long long key_tiles, long long tiles) { return key_tiles >= 3 * tiles; }

// The same with a cluster of 2^lg CTAs (or query heads folded, lg = 0): from four key tiles to a CTA on, below that the second warpgroup
// would only wait for its first scores (see FwdTmem in attn_fwd.cuh).
inline bool fwd_cluster_separate_rings(int key_tiles, int lg) { return (key_tiles >> lg) >= 4; }

// dQ side at d = 128: are the tiles so short that the compute warpgroups should prepare the row constants (SHORT in attn_bwd.cuh)?
// key_tiles, tiles: of one head.  Measured, off -> on, causal, rows (key tiles per tile): 256 (1.5) 162 -> 124 us, 500 (2.5) 371 -> 293, 700
// (3.5) 147 -> 133, 1000 (4.5) 83.3 -> 83.3, 2300 (9.5) 212 -> 219; not causal: 256 (2) 142 -> 125, 384 (3) 123 -> 125, 500 (4) 181 -> 192.
inline bool dq_short_tiles(long long key_tiles, long long tiles, bool causal) { return 2 * key_tiles <= (causal ? 7 : 5) * tiles; }

// CTAs per query tile of the forward (its base-two logarithm): with few tiles and long key ranges a tile's key range is
// split over a cluster of 2, 4 or 8 CTAs, as many as leave each of their two warpgroups at least two 128-key tiles and let
// all clusters run at once (`fit`: how many clusters of 2^lg CTAs do).  Beyond one wave the split only adds its merge.  Measured, one
// CTA per tile -> cluster, d = 64: 49 heads x 15 queries behind 17059 keys: 104 -> 59.3 us (two CTAs), 61 x 3 behind 6496: 42.6 ->
// 27.1, 17 x 128 behind 8346: 53.1 -> 25.2 (four); d = 128: 56.6 -> 27.5, 13 x 128 behind 13398: 94.2 -> 26.8 (eight).  At 7 to 12 key
// tiles it depends on the tiles: 64 x 128 behind 915: 10.6 -> 13.0, but 3 x 63 behind 1490: 13.0 -> 8.7 with eight CTAs and 16 x 1
// behind 842: 9.1 -> 7.4 with four, which the limit of 16 key tiles, as an older merge needed it, leaves out.
inline int fwd_cluster_log2(long long tiles, int key_tiles, const int (&fit)[4]) {
  int lg = 0;
  while (lg < 3 && key_tiles >= std::max(16, 4 << (lg + 1)) && tiles <= fit[lg + 1]) ++lg;
  return lg;
}

// Causal forward of grouped queries shorter than a tile: is it faster with the G query heads of a KV head folded into one head
// of G N rows?  Folded, the kernel runs one tile per CTA (or cluster) and merges its parts through shared memory, which costs
// more per tile than the persistent form; unfolded, every head is a tile of its own with N of its 128 rows in use.  The two
// times are estimated in microseconds from what was measured (148 CTAs at once):
//   folded          with u the share of the tile's rows in use: per round 5.7 + 2.25 u + (0.785 + 0.135 u) per key tile of a CTA at
//                   d = 64, less 0.35; 7.15 + 5 u + 1 per key tile, less 0.9, at d = 128.  Whole heads in clusters: the same
//   whole heads     d = 64: 3.1 + per round 1.1 + 0.765 per key tile; d = 128: 1.7 + per round 3.85 + 0.87 per key tile while the key
//                   range of a tile is split between the warpgroups; beyond 1.5 tiles per SM, where it is not, 2.1, 2.7, 1.82
// Folded also where the estimates are within 3 %: it reads the keys once, which a busy memory system rewards.  Never where whole
// heads are in clusters already and folding does not make the tiles fewer.
// Measured, whole -> folded, d = 64: 16 x (32 query, 8 KV heads) x 1 query behind 1000 keys: 32.7 -> 12.1 us; 64 x (32, 8) x 64
// behind 2048: 185 -> 159; but 32 x (64, 4) x 64 behind 600: 73.9 -> 90.9 and x 120: 74.6 -> 170; 64 x (16, 4) x 100 on as many keys:
// 18.3 -> 61.8; 2 x (64, 8) x 100 behind 1000: 11.0 -> 15.4.  d = 128: 70.4 -> 13.9, 447 -> 195, 172 -> 119; 182 -> 221, 36.1 -> 88.3,
// 13.7 -> 19.3.  Over 410 sizes that the figures were not fitted to, at both head dimensions, the choice costs 0.2 % on average
// against the better of the two, more than 3 % in 18 of the 820 and 17 % at most.
inline bool fwd_folds_heads(int kv_heads, int G, int N, int Nk, int d, int sms, const int (&fit)[4]) {
  if (N >= 128) return false;
  const bool wide = d == 128;
  const int key_tiles = (Nk + 127) / 128;
  const long long whole = static_cast<long long>(kv_heads) * G, folded = static_cast<long long>(kv_heads) * ((static_cast<long long>(G) * N + 127) / 128);
  auto rounds = [&](long long tiles) { return static_cast<double>((tiles + sms - 1) / sms); };
  auto merged = [&](long long tiles, long long rows) {
    const int lg = fwd_cluster_log2(tiles, key_tiles, fit);
    const double used = static_cast<double>(std::min<long long>(128, rows)) / 128;
    return (lg > 0 ? 1.0 : rounds(tiles)) * ((wide ? 7.15 + 5.0 * used : 5.7 + 2.25 * used) + (wide ? 1.0 : 0.785 + 0.135 * used) * ((key_tiles + (1 << lg) - 1) >> lg)) - (wide ? 0.9 : 0.35);
  };
  double t_whole;
  if (fwd_cluster_log2(whole, key_tiles, fit) > 0) {
    if (folded == whole) return false;
    t_whole = merged(whole, N);
  }
  else if (!wide) t_whole = 3.1 + rounds(whole) * (1.1 + 0.765 * key_tiles);
  else if (2 * whole < 3LL * sms) t_whole = 1.7 + rounds(whole) * (3.85 + 0.87 * key_tiles);
  else t_whole = 2.1 + rounds(whole) * (2.7 + 1.82 * key_tiles);
  return merged(folded, static_cast<long long>(G) * N) < 1.03 * t_whole;
}

// CTAs per (head, sequence) of key smoothing: 1, 2, 4 or 8.  pairs: (head, sequence) pairs of the launch; rows: their rows
// together; longest: rows of the longest one.  A pair is split further
//   - while all CTAs still run at once (three per SM: the fourth is there for uneven sequences), or
//   - while what the running pairs read is more than L2 holds until the second pass, or while a CTA of the longest sequence has
//     more than 1024 rows, which it alone would be busy with at the end;
// but not below 32 KB of a CTA's rows, nor beyond four unless few long sequences are all there is.
// Measured, CTAs per pair 8, 4, 2, 1 [taken], d = 64: 64 x 32 heads x 200: 249, 78, 37, [21] us; x 1000: 265, 118, [98], 113; x 2048: 308,
// [201], 231, 244; 4 x 32 x 4096: 39, [30], 32, 44; 16 x 4096: 9.5, [8.7], 13, 21; 4 x 8000: [9.1], 12.8, 22, 38.  d = 128: 64 x 32 x 512: 437, 135, [101],
// 116; 16 x 16 x 1000: 72, 35, 28, [30]; 24 documents, 19446 rows, 4 heads: 31, [19], 24, 30.
constexpr int kSmoothCtasPerSm = 4;
inline int smooth_cluster(long long pairs, long long rows, int longest, int d, int sms) {
  const int least = 32 * 1024 / (2 * d);               // rows of a CTA
  const double bytes = 2.0 * d * static_cast<double>(rows);
  int c = 1;
  while (c < 4 && longest >= 2 * c * least) {
    const double running = std::min(1.0, static_cast<double>(kSmoothCtasPerSm) * sms / c / static_cast<double>(pairs));
    if (pairs * 2 * c > 3LL * sms && running * bytes <= 70e6 && longest <= 1024 * c) break;
    c *= 2;
  }
  return c == 4 && longest > 4096 && pairs * 8 <= 3LL * sms ? 8 : c;
}

// The row offsets of a packed call (host).
struct PackedSeqs { const int *cu_q, *cu_k; int num; bool causal; };

// Work of every tile of a packed call, in the plan's order (decreasing): keys of each query tile (key_side: queries of each
// key tile, whose walk starts at a 64-row block).
inline std::vector<int> packed_work(const PackedSeqs &ps, bool key_side) {
  std::vector<int> work;
  for (int s = 0; s < ps.num; ++s) {
    const int lq = ps.cu_q[s + 1] - ps.cu_q[s], lk = ps.cu_k[s + 1] - ps.cu_k[s], off = lk - lq;
    if (!key_side)
      for (int r = 0; r < lq; r += 128) work.push_back(ps.causal ? std::max(0, std::min(lk, std::min(r + 128, lq) + off)) : lk);
    else if (lq > 0)
      for (int r = 0; r < lk; r += 128) work.push_back(std::max(0, lq - (ps.causal ? std::max(0, r - off) & ~63 : 0)));
  }
  std::sort(work.begin(), work.end(), [](int a, int b) { return a > b; });
  return work;
}

// Key tiles that a head's query tiles walk over all sequences.
inline long long walked_key_tiles(const PackedSeqs &ps) {
  long long sum = 0;
  for (int s = 0; s < ps.num; ++s) sum += fwd_key_tiles(ps.cu_q[s + 1] - ps.cu_q[s], ps.cu_k[s + 1] - ps.cu_k[s], ps.causal);
  return sum;
}

inline int longest_keys(const PackedSeqs &ps) {
  int most = 0;
  for (int s = 0; s < ps.num; ++s) most = std::max(most, ps.cu_k[s + 1] - ps.cu_k[s]);
  return most;
}

// What each CTA gets in the static deal (TileSched, walked item by item) of `items` items.  work_of is called once for every item, in order.
template <typename WorkOf>
std::vector<double> deal_loads(long long items, int ctas, WorkOf work_of, int solo = 0) {
  const int G = static_cast<int>(std::min<long long>(items, ctas)), W = G - solo;
  std::vector<double> load(static_cast<size_t>(G));
  long long lin = 0;
  for (int c = 0; c < G; ++c) load[static_cast<size_t>(c)] = work_of(lin++);
  for (bool odd = true; lin < items; odd = !odd) {
    const int n = static_cast<int>(std::min<long long>(W, items - lin));
    if (odd) for (int c = 0; c < n; ++c) load[static_cast<size_t>(G - 1 - c)] += work_of(lin++);
    else     for (int c = 0; c < n; ++c) load[static_cast<size_t>(solo + c)] += work_of(lin++);
  }
  return load;
}
// The longest of them.
template <typename WorkOf>
double deal_makespan(long long items, int ctas, WorkOf work_of, int solo = 0) {
  const std::vector<double> load = deal_loads(items, ctas, work_of, solo);
  return *std::max_element(load.begin(), load.end());
}

// ... of `heads` copies of every tile, with the cost that cost_of gives for its steps.
template <typename CostOf>
std::vector<double> deal_tile_loads(const std::vector<int> &steps, int heads, int ctas, CostOf cost_of, int solo = 0) {
  size_t k = 0;
  int left = 0;
  double cost = 0.0;
  return deal_loads(static_cast<long long>(steps.size()) * heads, ctas, [&](long long) {
    if (left == 0) { cost = cost_of(steps[k++]); left = heads; }
    --left;
    return cost;
  }, solo);
}
template <typename CostOf>
double deal_tiles(const std::vector<int> &steps, int heads, int ctas, CostOf cost_of, int solo = 0) {
  const std::vector<double> load = deal_tile_loads(steps, heads, ctas, cost_of, solo);
  return *std::max_element(load.begin(), load.end());
}

// fwd_separate_rings for a packed call of few items per CTA: what counts is the CTA that takes longest (its items' key tiles, and
// fwd_item_cost more for each), which has long tiles where the others have many short ones.  48 documents of 6288 rows together, 2 heads, causal: one
// ring 23.5 us, two 19.8; 49 pairs of 3485 queries and 13379 keys, 4 heads: 26.9, 23.1.
inline bool fwd_separate_rings(const std::vector<int> &key_tiles, int heads, int sms, int solo) {
  const double cost = fwd_item_cost(128, false);
  const std::vector<double> load = deal_tile_loads(key_tiles, heads, sms, [&](int n) { return n + cost; }, solo);
  const std::vector<double> items = deal_tile_loads(key_tiles, heads, sms, [](int) { return 1.0; }, solo);
  const size_t c = static_cast<size_t>(std::max_element(load.begin(), load.end()) - load.begin());
  return load[c] - cost * items[c] >= 3.0 * items[c] - 1e-6;
}

// TileSched's solo CTAs for `heads` copies of tiles with the given costs (decreasing): those whose first item is longer than
// what an even share of the rest would be.  The boustrophedon rounds would give each of them a second item all the same.
// Measured, 12 packed pairs (4000 queries, 9000 keys, 12 heads, d = 128; 60 of 456 query tiles twice as long as an even
// share): forward 53.6 -> 45.5 us, dQ side 76.5 -> 64.0 us.
// per_item: the kernel's measured overhead per item, in steps.
inline int solo_ctas(const std::vector<int> &steps, int heads, int sms, double per_item) {
  const long long items = static_cast<long long>(steps.size()) * heads;
  if (items <= sms || items > 16LL * sms) return 0;
  auto cost = [&](int n) { return n + per_item; };
  double rest = 0.0;
  for (int n : steps) rest += cost(n) * heads;
  int solo = 0;
  while (solo < sms / 2 && cost(steps[static_cast<size_t>(solo / heads)]) > rest / (sms - solo)) rest -= cost(steps[static_cast<size_t>(solo++ / heads)]);
  if (solo == 0) return 0;
  return deal_tiles(steps, heads, sms, cost, solo) < 0.99 * deal_tiles(steps, heads, sms, cost) ? solo : 0;
}

// Share every tile of a backward kernel between the two CTAs of a cluster?  This replays the static deal of both forms in
// units of one step (per_item: the kernel's measured overhead per item; exchange: what the exchange of the two parts adds)
// and takes the pairs where their longest CTA is 3 % shorter.  steps: of each tile of a head, decreasing.
// Measured, dK/dV side at d = 64 alone, whole tiles -> pairs: 16 query / 4 KV heads x 4096, causal: 121 -> 77 us; 8 / 2 heads x 8000,
// causal: 229 -> 140; 32 / 4 heads x 2000: 121 -> 78; 4 heads x 4096, causal: 43.5 -> 37.2; 1 head x 8192: 62.0 -> 43.5;
// 16 heads x 4096, causal (stays with whole tiles): 68; 16 packed documents of 8192 rows, 16 / 4 heads: 78.6 -> 73.0.
// dK/dV side at d = 128: 16 / 4 heads x 4096, causal: 275 -> 151; 8 / 1 heads x 3000, causal: 375 -> 200; 16 / 8 heads x 700, causal: 30.9 ->
// 25.0; 2 heads x 1500, causal: 30.9 -> 24.8; 4 heads x 1000 (16 steps): 24.7 -> 21.0; 4 heads x 800, causal: 20.7 -> 19.1; 2 heads x 640 (10
// steps): 17.5 -> 17.1, hence four steps for the exchange.
// dQ side: 1 head x 8192 x 64: 83 -> 52 us; 4 heads x 4096 x 64, causal: 44.7 -> 34.4; 16 heads x 300 queries behind 9000 keys,
// d = 128: 126 -> 92; 4 heads x 2048 x 128, causal: 36.5 -> 32.8; 4 heads x 1000 x 128 (16 steps): 20.7 -> 21.3, hence the
// 8 steps the exchange counts at d = 128.
inline bool prefers_pairs(const std::vector<int> &steps, int heads, int sms, int pairs, double per_item, double exchange) {
  const long long items = static_cast<long long>(heads) * static_cast<long long>(steps.size());
  if (pairs < 1 || items < 1 || items > 8LL * sms) return false;      // many items per CTA: they balance as they are
  const double whole = deal_tiles(steps, heads, sms, [&](int n) { return n + per_item; });
  const double split = deal_tiles(steps, heads, pairs, [&](int n) { return (n + 1) / 2 + per_item + exchange; });
  return split < 0.97 * whole;
}

// Steps of `rows` rows of the tiles of a call (key_side: of the key tiles, over the G heads of a group), decreasing.
inline std::vector<int> tile_steps(const PackedSeqs &seqs, bool key_side, int rows, int G) {
  std::vector<int> steps = packed_work(seqs, key_side);
  for (int &w : steps) w = G * std::max(1, (w + rows - 1) / rows);
  return steps;
}

// How the items of a backward kernel are dealt: every tile shared by two CTAs, or else `solo` CTAs with one item only.
struct DealForm { bool pairs; int solo; };
struct DealCosts { int rows; double per_item, exchange; };   // rows of a step; prefers_pairs
// tiles: of a head.  Beyond 16 items per CTA neither matters, and beyond 8 (where dense calls end, whose tiles need no solo CTAs) only
// solo: the tiles are not even listed (8000 packed sequences: 120 us of host time).
inline DealForm deal_form(const PackedSeqs &seqs, bool packed, bool key_side, int G, int heads, int tiles, int sms, int fit, const DealCosts &c) {
  const long long items = static_cast<long long>(heads) * tiles;
  if (items < 1 || items > (packed ? 16LL : 8LL) * sms) return DealForm{false, 0};
  const std::vector<int> steps = tile_steps(seqs, key_side, c.rows, G);
  if (prefers_pairs(steps, heads, sms, fit, c.per_item, c.exchange)) return DealForm{true, 0};
  return DealForm{false, packed ? solo_ctas(steps, heads, sms, c.per_item) : 0};
}

}  // namespace gproj
