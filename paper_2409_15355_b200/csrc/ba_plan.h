// How the attention launches are laid out: host arithmetic on plain numbers, no device and no CUDA headers.
#pragma once

#include <algorithm>
#include <stdint.h>

// How ba_final_attend divides the key tiles of its work items among CTAs (pure host arithmetic, also reachable
// through ba_plan_final_attend).  Inputs: SMs; work items (query tile pairs x head chunks); pairs and head chunks;
// key tiles of an average item; sum / minimum / maximum of the key tiles over the pairs when known (else zeros);
// the most partial results per row the workspace has room for.
//  * Equal splits: n_splits entries per item, the count that minimises waves x (tiles per entry + 3), the 3
//    standing for an entry's start-up and write-out.
//  * Balanced launch (item sizes known, fewer items than SMs, every item longer than an SM's share of the tiles):
//    one CTA per item takes the item's last `len` key tiles, the remaining CTAs share the tiles in front of those
//    in equal runs.  `len` starts at the even share and grows until the CTAs that work on several pieces (each
//    with its own start-up and write-out, plus 1 for their table) are no longer the slower ones.  Taken when the
//    same cost model puts it ahead of equal splits; n_splits is then the number of partial results per row.
constexpr int kBalMaxPairs = 120;        // the balanced launch keeps a prefix table of this many pairs in shared memory
struct ba_split_plan { int n_splits, balanced, bal_len; };
static inline ba_split_plan ba_plan_splits(int sm_count, long long items, int n_pairs, int n_chunks, long long avg_tiles,
                                           const int32_t *key_tiles, int cap) {
  ba_split_plan plan = {1, 0, 0};
  if (items >= 2LL * sm_count || cap < 1) return plan;
  long long best = -1;
  for (int ns = 1; ns <= cap && ns <= avg_tiles; ++ns) {
    const long long waves = (items * ns + sm_count - 1) / sm_count;
    const long long cost = waves * ((avg_tiles + ns - 1) / ns + 3);
    if (best < 0 || cost < best) { best = cost; plan.n_splits = ns; }
  }
  const long long n_main = (long long)n_pairs * n_chunks;
  const long long n_front = sm_count - n_main;
  if (key_tiles[0] > 0 && n_main > 0 && n_front > 0 && n_pairs <= kBalMaxPairs) {
    const long long total = (long long)key_tiles[0] * n_chunks, n_min = key_tiles[1], n_max = key_tiles[2];
    for (long long len = (total + sm_count - 1) / sm_count; len <= n_min; ++len) {
      const long long front = total - n_main * len;
      if (front <= 0) break;
      const long long run = (front + n_front - 1) / n_front, run_min = front / n_front;
      if (run_min < 1) break;
      const long long piece = (front + n_main - 1) / n_main;          // average front tiles of an item
      const long long cost_front = run + 3 * ((run + piece - 1) / piece + 1) + 1;
      if (cost_front > len + 3) continue;
      const long long slots = 1 + (n_max - len + run_min - 1) / run_min + 1;
      if (len + 3 < best && slots <= cap) { plan.balanced = (int)n_main; plan.bal_len = (int)len; plan.n_splits = (int)slots; }
      break;
    }
  }
  return plan;
}

// Time of equal splits in key tiles (an entry's start-up and write-out count as 3, the merging kernel as 5); every wave is
// as long as its longest entry.
static inline long long ba_equal_splits_cost(int sm_count, long long items, long long max_tiles, int n_splits) {
  const long long waves = (items * n_splits + sm_count - 1) / sm_count;
  return waves * ((max_tiles + n_splits - 1) / n_splits + 3) + (n_splits > 1 ? 5 : 0);
}

// Stream launch of ba_final_attend: the key tiles of all items, end to end, in one run per CTA.  Each CTA works on about
// 1 + run / item pieces of items; a piece that is not a whole item costs a partial result.  There are two such streams, one
// of every sequence's items 0, 2, .. and one of its items 1, 3, .. (n_odd of the CTAs).  key_tiles: sum, minimum, maximum
// over the items of one head chunk, odd_tiles: sum over the second stream.  cap: the most partial results per row.
struct ba_stream_plan { int n_ctas, n_odd, n_slots; long long cost; };
static inline ba_stream_plan ba_plan_stream(int sm_count, int n_chunks, const int32_t *key_tiles, int odd_tiles, int cap) {
  ba_stream_plan plan = {0, 0, 0, 0};
  const long long total = (long long)key_tiles[0] * n_chunks, odd = (long long)odd_tiles * n_chunks, n_max = key_tiles[2];
  if (total <= 0 || total > 0x3fffffff) return plan;
  const long long g = total < 2LL * sm_count ? (total + 1) / 2 : sm_count;
  // the division of the CTAs that leaves the shorter longest run; a stream in one run has no cuts
  long long run = total + 1, run_min = total, n_odd = 0;
  for (long long n = odd * g / total; n <= odd * g / total + 1; ++n) {
    if (n >= g || (n == 0) != (odd == 0)) continue;
    const long long even = total - odd, e = g - n;
    const long long longest = std::max((even + e - 1) / e, n ? (odd + n - 1) / n : 0);
    if (longest >= run) continue;
    run = longest; n_odd = n;
    run_min = std::min(e > 1 ? even / e : total, n > 1 ? odd / n : total);
  }
  if (run > total || (run == total && g > 1)) return plan;   // no division gives each stream that has tiles a CTA; no gain
  const long long slots = (n_max - 1) / std::max(run_min, 1LL) + 2;   // runs an item of n_max tiles can touch
  if (slots > cap) return plan;
  const long long pieces = 1 + (run + n_max - 1) / n_max;
  plan.n_ctas = (int)g; plan.n_odd = (int)n_odd; plan.n_slots = (int)slots; plan.cost = run + 2 + 2 * pieces + 5;
  return plan;
}

// Cluster launch of ba_final_attend: the `size` CTAs of a cluster share one item's key tiles and merge their results in
// shared memory, which saves the partial results' way through memory and the merging kernel.  single: a cluster takes one query
// tile of an item instead of two, where most items have two (`two_tiles`): a CTA has half the rows to fetch, write out and collect
// from the others.  shared: every CTA has one query tile (one_tile: no item has two), and unless the call is the fused one both softmax
// groups share its key tiles.  A CTA's time in key tiles of two query tiles, its start and write-out, and the merge:
//   two query tiles, or one of a whole item     1    a tile, 3,   1.5
//   one query tile, fused                       0.85 a tile, 3,   0.25
//   one query tile, shared by both groups       0.6  a tile, 3.5, 0.25
// The last row was fitted to 240 shapes of 1-8 requests, 16-256 final and 250-9000 cached tokens, six shapes of heads, every layout and
// cluster size timed (32/8 heads, us a launch, whole items, single tiles, no cluster: 6000 cached tokens and 64 final ones 24.6, 19.8, 23.1;
// 128 final ones 28.5, 23.8, 25.8; 1000 and 256 20.1, 18.5, 20.1).  With the prices from before the groups shared tiles (the second row and,
// for items of one tile, the first) 30 of them took a layout that is 0.6-19 % slower (6000 and 128: whole items; two requests
// of 9000 and 20: 28.9 us without a cluster, 23.5 with), none a faster one.  Sharing is not for CTAs with two query tiles, where that
// kernel is the slower one: with a re-encoding pass, 6000 cached tokens and 65 / 128 / 256 final ones 35.8 and 36.5, 36.9 and 37.6,
// 45.7 and 47.0; four requests of 6000 and 8, 8, 8 and 60 55.2 and 56.4.  fits(size): clusters of that size the GPU runs at a time
// (0: none).
constexpr int kMaxCluster = 8;
struct ba_cluster_plan { int size, single, shared; double cost; };
template <class Fits>
static inline ba_cluster_plan ba_plan_cluster(long long items, bool two_tiles, bool one_tile, bool fused, long long max_tiles, Fits fits) {
  ba_cluster_plan plan = {0, 0, 0, 0.};
  for (int single = 0; single <= (two_tiles ? 1 : 0); ++single)
    for (int n = 2; n <= kMaxCluster && n <= max_tiles; ++n) {
      const long long units = items << single, at_a_time = units == 1 ? 1 : fits(n);
      if (at_a_time < 1) continue;
      const bool shared = !fused && (single || one_tile);
      const double tile = shared ? 0.6 : single ? 0.85 : 1.0, start = shared ? 3.5 : 3.0, merge = shared || single ? 0.25 : 1.5;
      const double cost = (double)((units + at_a_time - 1) / at_a_time) * ((max_tiles + n - 1) / n * tile + start) + merge;
      if (!plan.size || cost < plan.cost) { plan.size = n; plan.single = single; plan.shared = shared; plan.cost = cost; }
    }
  return plan;
}

// ba_block_prefill in block mode: into how many pieces the key tiles of a final block's items are cut, so that no entry is
// longer than half of what an SM gets altogether (an entry's start-up and write-out count as one tile in a full list).
static inline int ba_plan_final_splits(int sm_count, int n_chunks, int n_items, int n_tiles, int longest, int cap) {
  const long long share = ((long long)n_tiles + n_items) * n_chunks / sm_count;
  const long long piece = share / 2 > 6 ? share / 2 : 6;
  const long long want = (longest + piece - 1) / piece;
  return (int)(want < 1 || cap < 2 ? 1 : want < cap ? want : cap);
}
