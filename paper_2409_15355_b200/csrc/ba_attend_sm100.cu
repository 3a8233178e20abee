// Tensor-core attention under the Block-attention mask for sm_100a.
//
// One kernel serves ba_block_prefill (Section 1 / 2.4: a row of a non-final block
// sees its own block, causally; a row of a final block sees its whole sequence
// prefix) and ba_final_attend (Section 2.5 step 3: the final block over the
// re-encoded cached blocks plus itself).  The mask never exists as a matrix: a
// work item is a pair of query tiles of one block, its keys are one optional
// "cached" range (all visible) followed by one "own" range (causal).
//
// Structure of a CTA (384 threads, one CTA per SM):
//   warps 0-3   softmax of query tile 0      (one thread per tile row = TMEM lane)
//   warps 4-7   softmax of query tile 1 (kSharedCluster, where there is one query tile only: of every second key tile)
//   warp  8     TMA producer: Q tiles once, then K_j, V_j, K_j+1, ... into a ring of stages (key tiles shared by both softmax
//               groups: K_0, K_1, V_0, K_2, V_1, ...)
//   warp  9     MMA issuer (one elected thread): S = Q K^T and O += P V with tcgen05.mma,
//               accumulators in tensor memory (S0, S1, O0, O1 = 4 x 128 columns)
// A query tile is 128 rows = (128 / HPT) tokens x HPT query heads of one KV group,
// so a K/V tile staged once serves every head of the group and both query tiles.
// Softmax is online in fp32 (base-2 exponent with the scale folded in); P is
// written back to tensor memory as bf16 over the S columns and used as the A
// operand of the PV product.  O is rescaled in tensor memory only when the
// running maximum grows by more than 2^8, which keeps every term bounded and the
// result exact in real arithmetic.
//
// Fused warm path (Section 2.5 steps 2 and 3 in one launch): the cached keys stay at their
// cache-time positions and the position difference of each block (Eq. 3 after Eq. 2) is applied
// to the other side of the dot product, (R(p) q) . (R(delta + t) k) = (R(-delta) R(p) q) . (R(t) k):
// each softmax thread owns one row of its query tile and prepares, for every cached block of the
// work entry, a copy of that row rotated by the block's delta (and a plain copy for the final
// block's own keys) in one of two buffers per query tile.  The copy for the next block is made
// while the current block's tiles are worked on -- the plain tile is fetched after one tile and
// rotated in place after the next, in time the thread would otherwise spend waiting for S --
// so the QK^T products switch buffers without a pause.  The cached keys are never rewritten or
// re-read, and a key tile never spans two blocks.
#include <math.h>
#include <atomic>
#include <new>
#include <type_traits>

#include "ba_common.cuh"
#include "ba_sm100.cuh"
#include "ba_reencode_dev.cuh"

using namespace sm100;

// Tuning aid, absent from ordinary builds: with -DBA_TRACE the roles of CTA 0 stamp clock64() at the
// phases of their first 64 key tiles into a device array that a developer build reads back
// (roles 0/1: softmax groups, 2: MMA thread per query tile, 3: MMA thread's K/V waits, 5: fused query versions).
#ifdef BA_TRACE
__device__ long long g_ba_trace[6][64][8];
extern "C" int ba_trace_read(long long *dst) { return (int)cudaMemcpyFromSymbol(dst, g_ba_trace, sizeof(g_ba_trace)); }
#define BA_TR(role, tile, k)                                                                  \
  do {                                                                                        \
    if (blockIdx.x == 0 && (tile) < 64) g_ba_trace[role][tile][k] = clock64(); \
  } while (0)
#else
#define BA_TR(role, tile, k) do { } while (0)
#endif

namespace {

constexpr int kThreads = 384;
constexpr int kBlockN = 128;      // keys per tile
// Variants of the kernel, so that each carries only its own code.  The ring of K/V tiles (K_j, V_j, K_j+1, ...; in kSharedCluster
// K_0, K_1, V_0, K_2, V_1, ...) has three stages; the rest of the shared memory is a second pair of query buffers (or the
// background job's staging area).  In kDeepRing it is a fourth stage and a staging area for the write-out: a tile that comes from
// HBM while every SM streams takes 2000-4500 cycles, three stages cover 2700 (64-token query over 32K cached keys: 800-1900 cycles
// of waiting in a period of 4000-4900; with four the product thread finds every tile there), and with the write-out elsewhere the
// one pair of query buffers is reloaded as soon as its last product is done.
// The cluster forms of the last two merge the results of a cluster's CTAs in shared memory; kSharedCluster is kDeepCluster for
// launches whose CTAs have one query tile (is_solo).
constexpr int kPlain = 0, kFusedPath = 1, kDeepRing = 2, kFusedCluster = 3, kDeepCluster = 4, kSharedCluster = 5;
constexpr bool is_fused(int variant) { return variant == kFusedPath || variant == kFusedCluster; }
constexpr bool is_deep(int variant) { return variant == kDeepRing || variant == kDeepCluster || variant == kSharedCluster; }
constexpr int kMaxStages = 4;
constexpr float kRescaleThreshold = 8.0f;
constexpr int kBgStageBytes = 16384; // two spare warps x two stages of source rows
constexpr int kWorkSlots = 4;      // ring of published work entries (power of two)
constexpr int kBalTableOff = 512;  // balanced launch: prefix table of front tiles, in the control area behind Ctrl
// (its capacity, kBalMaxPairs items per head chunk, is declared with the planning arithmetic; the spare warps' barriers follow at 1024)
// Register split after launch (168 per thread): the service warps give registers to the softmax warps.
// 128 * kServiceRegs + 256 * kSoftmaxRegs <= 384 * 168.  The MMA thread keeps a work entry, descriptors
// and ring positions live and spills below about 88; the softmax warps start to spill below 208.  On the
// fused path the softmax warps also prepare query versions and need the larger share.
constexpr int kServiceRegsPlain = 88, kSoftmaxRegsPlain = 208;
constexpr int kServiceRegsFused = 72, kSoftmaxRegsFused = 216;

struct AttnParams {
  void *o;
  float *lse;
  int32_t *status;
  int out_f32;
  int Hq, Hkv, G;
  int hpt, hpt_log2, tok;         // heads per tile, tokens per tile (hpt * tok = 128)
  float scale, scale_log2;
  int final_only;
  int n_q_rows;
  int n_chunks;                   // head chunks per token (Hq / hpt)
  int n_splits;                   // > 1: the key tiles of an item are divided among several work entries, combined later
                                  // (prefill: of the items of final blocks only)
  float *o_part;                  // [n_splits, n_part_rows, Hq, D] fp32, each normalised by its own denominator
  float *lse_part;                // [n_splits, n_part_rows, Hq] natural-log denominators (-inf: split saw no key)
  int n_part_rows;
  // stream = 1: the key tiles of all (item, head chunk) are laid end to end and cut into one run per CTA, those of the
  // items 1, 3, .. of every sequence on the last n_odd CTAs
  int stream, n_odd;
  // cluster > 1: the CTAs of a cluster share one item's key tiles and merge their results in shared memory; single: one
  // query tile of an item
  int cluster, single;
  const int32_t *v_src_off;       // non-null: values of cached block c start at pool row v_src_off[c]
  int persistent;                 // 1: CTAs draw work from counters[0]; 0: CTA b handles entry b only
  // balanced > 0 (final block over a long cache, fewer items than CTAs): the first `balanced` CTAs each take the
  // last bal_len key tiles of one item (slot 0 of its partial results); the other CTAs share the key tiles in
  // front of those, cut into equal runs whatever item they fall in (slots 1 ..).  n_splits is the slot count.
  int balanced, bal_len;
  int q_double;                   // plain path, no background job: two pairs of query buffers (see Ctrl)
  // three device words, zero at launch and zero again when the launch ends (its last CTA clears them):
  // [0] next entry of the work list, [1] next chunk of the background job, [2] CTAs that have finished
  int32_t *counters;
  ba_reencode_job bg;             // bg.n_rows > 0: a re-encoding job the two spare warps carry out meanwhile
  int bg_rows_per_chunk;
  ba_segments seg;
  const int32_t *items;           // work items of this call (seg.final_items or seg.prompt_items)
  const int32_t *k_src_off;       // non-null: keys of cached block c start at pool row k_src_off[c] (fused path only)
  int walk;                       // cached keys are walked block by block (a tile never spans two blocks)
  // paged pool: cached block c owns the pages page_idx[page_cu[c] .. page_cu[c+1]) of 1 << page_lg rows each;
  // row t of the block is row t & (page_rows - 1) of page t >> page_lg of its list.  Applies to the values
  // (v_paged) and, on the fused path, to the keys (k_paged).
  const int32_t *page_cu, *page_idx;
  int page_lg, k_paged, v_paged;
  int fused;                      // cached keys are at cache-time positions: queries are counter-rotated per block
  int rope_layout;
  const float2 *q_rope;           // fused: [cached blocks][D/2] (cos, sin) of delta_c * theta_m
};

template <int D>
struct Layout {
  static constexpr int kChunks = D / 64;                  // 64-column (128-byte) swizzle regions per row
  static constexpr int kTileBytes = 128 * D * 2;          // one 128-row tile of Q, K or V
  static constexpr int kRegionBytes = 128 * 128;          // 128 rows x 128 bytes
  static constexpr int kQ0 = 0;
  static constexpr int kQ1 = kTileBytes;
  static constexpr int kRing = 2 * kTileBytes;
  static constexpr int kBg = kRing + 3 * kTileBytes;           // staging of the background re-encoding, the second pair
                                                               // of query tile buffers, or a fourth stage and staging rows
  static constexpr int kCtrl = kBg + 4 * kBgStageBytes;        // 2 KB: Ctrl, then two ba_bg_smem
  static constexpr int kBytes = kCtrl + 2048;
  static_assert(2 * kTileBytes <= 4 * kBgStageBytes, "two tiles fit the staging area");
};

// In lse_part (stream launch): the row needed no partial results, its output is written.  A NaN no arithmetic produces.
constexpr uint32_t kRowIsComplete = 0xffc0ba11u;

// What the scheduling thread publishes to the other roles of its CTA.
struct WorkEntry {
  int pair;            // item (index into the list of query tile pairs); < 0: no more work
  int chunk;           // head chunk
  int tile0, n_tiles;  // key tiles [tile0, tile0 + n_tiles) of the item
  int split;           // slot of the partial results this entry writes; < 0: it covers the whole item, rows go to the output
  int fill;            // slots fill .. n_splits - 1 of the item stay unused: this entry marks them empty (clusters: narrow_item)
};

struct Ctrl {
  // [buffer pair][query tile].  Plain path without a background job: the query tiles of successive entries
  // alternate between two pairs of buffers, so the next entry's queries are fetched while the current one runs.
  uint64_t q_full[2][2];
  // the buffer may be reloaded: the softmax warps have written the entry's rows out, which pass through it (kDeepRing: every
  // QK^T of the entry has completed, [0][0] only)
  uint64_t q_empty[2][2];
  uint64_t kv_full[kMaxStages];
  uint64_t kv_empty[kMaxStages];
  uint64_t s_full[2];
  uint64_t p_full[2][2];          // [query tile][half of the P tile]
  uint64_t o_done[2];
  uint64_t o_free[2];             // the softmax warps have read O_t out of tensor memory
  uint64_t out_staged[2];         // every row of the output tile is in shared memory
  uint64_t solo_full;             // one query tile, both softmax groups: group 1's maxima and sums are in shared memory
  int n_staged_out[2];            // output tiles handed to the copy engine so far
  uint64_t work_full[kWorkSlots];  // work entry published by the scheduler (producer thread)
  uint64_t work_empty[kWorkSlots]; // entry read by the MMA thread and the 8 softmax warps
  WorkEntry work_ring[kWorkSlots];
  int tile_valid[8];              // pool mode: valid key columns of the cached tiles in flight
  uint32_t tmem_base;
  int abort_flag;
  uint64_t qr_full[2][2];         // fused: [query tile][buffer] the tile prepared for the next key range is ready
  uint64_t cs_full[2];            // fused: the block's (cos, sin) row has been staged for softmax group t
  uint64_t qraw_full[2];          // fused: the plain query tile t has landed in the buffer of the version being prepared
};
static_assert(sizeof(Ctrl) <= kBalTableOff && kBalTableOff + (kBalMaxPairs + 1) * 4 <= 1024, "control area layout");

// One work item: two query tiles of one block (or final block) and the key ranges they see.
struct Item {
  int q_row0;        // first query row (q packing)
  int q_rows;        // valid query rows in the pair (1 .. 2*tok)
  int n_qt;          // 1 or 2 query tiles in use
  int cache_row0, cache_len;   // cached keys (cache packing), all visible
  int own_row0;      // first own key row (q packing); row i sees own rows own_row0 .. i
  int n_cache_tiles, n_tiles;
  int cb0;           // index (cache order) of the sequence's first cached block
  int ctile0;        // cache_tile_cu[cb0]: pool mode walks cached keys block by block
};

__device__ __forceinline__ float max3(float a, float b, float c) {
  float d;
  asm("max.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
  return d;
}

// The thread index, read where it is used: addresses that depend on it alone would otherwise be computed once and kept in
// registers through the softmax loop, which spills.
__device__ __forceinline__ int thread_index_anew() {
  int i;
  asm volatile("mov.u32 %0, %%tid.x;" : "=r"(i));
  return i;
}

// Work items of the call, as ba_segment left them (0 when the tables are not valid).
__device__ __forceinline__ int count_items(const AttnParams &p) {
  if (__ldg(p.seg.totals + 7) != BA_TABLES_VALID) return 0;
  return __ldg(p.seg.totals + (p.final_only ? 3 : 2));
}

// Partial results of a prefill are indexed by the row's place among the rows of final blocks, of which the host made room for
// n_part_rows; the tables may have been rebuilt in their buffer since.  (Those of a final attend are indexed by the query row.)
__device__ __forceinline__ bool partials_fit(const int32_t *totals, int final_only, int n_splits, int n_part_rows) {
  return final_only || n_splits <= 1 || __ldg(totals + 1) <= n_part_rows;
}

// Item `idx`: independent loads of one line of the table ba_segment built, instead of a search for the item's sequence or
// block and look-ups that depend on it.  (Four-byte loads: 16-byte ones tie up groups of four registers, and the softmax
// loop of the fused path spills.)
__device__ __forceinline__ void load_item(const AttnParams &p, int idx, Item &it) {
  const int32_t *x = p.items + 8 * (size_t)idx;
  it.q_row0 = __ldg(x); it.q_rows = __ldg(x + 1); it.own_row0 = __ldg(x + 2); it.cache_row0 = __ldg(x + 3);
  it.cache_len = __ldg(x + 4); it.cb0 = __ldg(x + 5); it.ctile0 = __ldg(x + 6);
  it.n_cache_tiles = p.walk ? __ldg(x + 7) : (it.cache_len + kBlockN - 1) / kBlockN;
  it.n_qt = it.q_rows > p.tok ? 2 : 1;
  it.n_tiles = it.n_cache_tiles + (it.q_row0 + it.q_rows - it.own_row0 + kBlockN - 1) / kBlockN;
}

// The part of its item that a cluster's entry covers (WorkEntry::fill: 1 + query tile, 0 the whole item).
__device__ __forceinline__ void narrow_item(const AttnParams &p, int fill, Item &it) {
  if (fill == 0) return;
  const int skip = (fill - 1) * p.tok;
  it.q_row0 += skip;
  it.q_rows = min(it.q_rows - skip, p.tok);
  it.n_qt = 1;
  it.n_tiles = it.n_cache_tiles + (it.q_row0 + it.q_rows - it.own_row0 + kBlockN - 1) / kBlockN;
}

// One entry of a CTA's work list: an item, the heads it covers and its share of the key tiles.
struct Work {
  Item it;
  int head0, kv_head;
  int tile0, n_tiles;   // key tiles [tile0, tile0 + n_tiles) of the item (split-KV share)
};

// The item of a published entry, decoded by the producer a few tiles ahead, for the roles whose wait for the item's line would stand
// between two entries (seven edited blocks, 312 entries, us over eight layers: 213 -> 209.5; cold prompt of 7200 tokens 784 -> 778).
struct ReadyItem { int q_row0, q_rows, own_row0, cache_len, n_cache_tiles, n_tiles, ctile0, pad; };
constexpr int kReadyOff = 1600;          // [kWorkSlots], in the control area behind the spare warps' barriers
static_assert(kReadyOff >= 1024 + 2 * (int)sizeof(ba_bg_smem) && kReadyOff + kWorkSlots * (int)sizeof(ReadyItem) <= 2048, "control area layout");
__device__ __forceinline__ bool ready_work(const AttnParams &p, const WorkEntry &e, const ReadyItem &x, Work &wk) {
  if (e.pair < 0) return false;
  wk.it.q_row0 = x.q_row0; wk.it.q_rows = x.q_rows; wk.it.own_row0 = x.own_row0; wk.it.cache_len = x.cache_len;
  wk.it.n_cache_tiles = x.n_cache_tiles; wk.it.n_tiles = x.n_tiles; wk.it.ctile0 = x.ctile0;
  wk.it.n_qt = x.q_rows > p.tok ? 2 : 1;
  wk.head0 = e.chunk * p.hpt;
  wk.tile0 = e.tile0;
  wk.n_tiles = e.n_tiles;
  return true;
}

// Cluster launch, an entry of one query tile: the two softmax groups share its key tiles.  Group 0 takes tiles 0, 2, .. and group
// 1 tiles 1, 3, .. with maxima, sums and an accumulator of its own (O_1), which group 0 merges when it writes the rows out.  One
// group alone leaves the tensor core idle while it exponentiates and the exponentials idle while the products run.  The ring then
// holds the keys one tile further ahead of the values: K_0, K_1, V_0, K_2, V_1, ..  (2500 cached tokens and a question of 64, 32
// layers: 706 -> 664 us.)  The test for it costs where there are two query tiles, as the thread that issues the products is on every
// tile's path: 16 pooled requests +5 %; clusters of whole items +1-3 % (ba_cluster_plan::shared: a kernel of their own without
// it).  At twice the keys per unit of time a ring of three stages runs dry: cold prompt of 7200 tokens 785 -> 890 us.
template <bool kAllowed>
__device__ __forceinline__ bool is_solo(const Work &wk) { return kAllowed && wk.it.n_qt == 1 && wk.n_tiles > 1; }

// Entry w of the global work list (equal shares of every item's key tiles).  pair < 0 past the end.
//  Prefill: items heaviest-first (descending index: the table ends with the items of the final blocks, and within a
//  sequence an item's cost grows with its index), then head chunk, then split (final blocks only).
//  Final attend: all items cost about the same, so the pair index varies fastest instead: the
//  CTAs running at the same time then work on the same (KV head, key range) for different query
//  tiles and each K/V tile comes from HBM once and from L2 for the others.
//  Clusters: the CTAs of a cluster are the splits of one item (p.single: of one query tile of it).
__device__ __forceinline__ WorkEntry cluster_entry(const AttnParams &p, int total_pairs) {
  WorkEntry e = {-1, 0, 0, 0, -1, 0};
  if (total_pairs <= 0) return e;
  const unsigned units = (unsigned)total_pairs << p.single, i = cluster_index(), chunk = i / units, rank = i - chunk * units;
  const unsigned k = cluster_rank(), n = (unsigned)p.cluster;
  if ((int)chunk >= p.n_chunks) return e;
  const int pair = total_pairs - 1 - (int)(rank >> p.single), fill = p.single ? 1 + (int)(rank & 1) : 0;
  Item it;
  load_item(p, pair, it);
  if (fill == 2 && it.n_qt < 2) return e;                  // (every CTA of the cluster leaves)
  narrow_item(p, fill, it);
  e.pair = pair; e.chunk = (int)chunk; e.split = (int)k; e.fill = fill;
  e.tile0 = (int)((unsigned)it.n_tiles * k / n);           // (at most 2^24 tiles, eight CTAs)
  e.n_tiles = (int)((unsigned)it.n_tiles * (k + 1) / n) - e.tile0;
  return e;
}
__device__ __forceinline__ WorkEntry list_entry(const AttnParams &p, int total_pairs, int w) {
  WorkEntry e = {-1, 0, 0, 0, -1, 0};
  int n_splits = p.n_splits, per_pair = p.n_chunks * n_splits, rank, rem;
  if (total_pairs <= 0) return e;
  if (p.final_only) {
    rem = w / total_pairs; rank = w - rem * total_pairs;
    if (rem >= per_pair) return e;
  } else {
    rank = 0;
    if (n_splits > 1) {                                    // first the items of final blocks, in pieces
      const int n_final = __ldg(p.seg.totals + 3);
      if (w >= n_final * per_pair) { w -= n_final * per_pair; rank = n_final; n_splits = 1; per_pair = p.n_chunks; }
    }
    rank += w / per_pair; rem = w % per_pair;
    if (rank >= total_pairs) return e;
  }
  Item it;
  e.pair = total_pairs - 1 - rank;
  load_item(p, e.pair, it);
  e.chunk = rem / n_splits;
  const int k = rem - e.chunk * n_splits;
  e.split = n_splits > 1 ? k : -1;
  e.fill = n_splits;
  e.tile0 = (int)(((long long)it.n_tiles * k) / n_splits);
  e.n_tiles = (int)(((long long)it.n_tiles * (k + 1)) / n_splits) - e.tile0;
  return e;
}

// A published entry, decoded by the role that reads it.  Returns false at the end of the work.
template <bool kClustered>
__device__ __forceinline__ bool load_work(const AttnParams &p, const WorkEntry &e, Work &wk) {
  if (e.pair < 0) return false;
  load_item(p, e.pair, wk.it);
  if (kClustered) narrow_item(p, e.fill, wk.it);
  wk.head0 = e.chunk * p.hpt;
  wk.kv_head = wk.head0 / p.G;
  wk.tile0 = e.tile0;
  wk.n_tiles = e.n_tiles;
  return true;
}

// Stream launch.  The key tiles of all (sequence, head chunk, item), in that order, are laid end to end and cut into one
// run per CTA, so that every SM gets the same number of tiles whatever the items' number and sizes.  A cut within
// kStreamSnap tiles of an item's edge is moved to the edge: a sliver of an item costs more than its tiles.
// There are two streams, one of every sequence's items 0, 2, .. and one of its items 1, 3, .., each on CTAs of its own: two
// successive items of a sequence read the same keys, and the two streams get to them at the same time, so that one of
// them finds them in L2.  (In one stream the second item comes a whole item later, when every SM has read some 50 tiles
// of 64 KB since: 16 requests of 20 cached blocks of 50-500 tokens, 128 final tokens, four layers, 1333 us, now 1284.)
constexpr int kStreamSnap = 2;
struct StreamState {
  int pos, end;              // tiles left to this CTA: [pos, end)
  int seq, chunk, i;         // item i of sequence seq that holds pos, its first tile g0
  int g0, cached_tiles, final_rows, n_items, item0;
  int total;
};
__device__ __forceinline__ void stream_sequence(const AttnParams &p, StreamState &s) {
  const int32_t *ft = p.seg.cu_ftile + s.seq, *fs = p.seg.cu_final_seq + s.seq;
  s.item0 = __ldg(ft); s.n_items = __ldg(ft + 1) - s.item0;
  s.final_rows = __ldg(fs + 1) - __ldg(fs);
  Item it;
  load_item(p, s.item0, it);
  s.cached_tiles = it.n_cache_tiles;
}
__device__ __forceinline__ int stream_item_tiles(const AttnParams &p, const StreamState &s) {
  return s.cached_tiles + (min((s.i + 1) * 2 * p.tok, s.final_rows) + kBlockN - 1) / kBlockN;
}
// This CTA's stream, its place among the CTAs of it and their number.
__device__ __forceinline__ int stream_of(const AttnParams &p) { return blockIdx.x >= gridDim.x - p.n_odd; }
__device__ __forceinline__ int stream_cta(const AttnParams &p) { return (int)(stream_of(p) ? blockIdx.x - (gridDim.x - p.n_odd) : blockIdx.x); }
__device__ __forceinline__ int stream_ctas(const AttnParams &p) { return stream_of(p) ? p.n_odd : (int)gridDim.x - p.n_odd; }
// Tiles of stream `lane`, one head chunk, in front of a sequence.
__device__ __forceinline__ int stream_before(const AttnParams &p, int lane, int seq) {
  const int32_t *cu = p.seg.cu_stream + (p.walk ? p.seg.batch + 1 : 0) + seq;
  const int odd = __ldg(cu + 2 * (p.seg.batch + 1));
  return lane ? odd : __ldg(cu) - odd;
}
// The item that holds tile x.
__device__ __forceinline__ void stream_locate(const AttnParams &p, StreamState &s, int x) {
  int lo = 0, hi = p.seg.batch - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (stream_before(p, stream_of(p), mid) * p.n_chunks <= x) lo = mid; else hi = mid - 1;
  }
  s.seq = lo;
  const int first = stream_before(p, stream_of(p), lo), per_chunk = stream_before(p, stream_of(p), lo + 1) - first;
  int r = x - first * p.n_chunks;
  s.chunk = r / per_chunk;
  r -= s.chunk * per_chunk;
  s.g0 = x - r;
  stream_sequence(p, s);
  s.i = stream_of(p);
  for (int n; r >= (n = stream_item_tiles(p, s)) && s.i + 2 < s.n_items; s.i += 2) { r -= n; s.g0 += n; }
}
// This CTA's run (all lanes of a warp).
__device__ __forceinline__ void stream_start(const AttnParams &p, StreamState &s) {
  s.total = stream_before(p, stream_of(p), p.seg.batch) * p.n_chunks;
  const int lane = threadIdx.x & 31;
  const int x = (int)((long long)s.total * (stream_cta(p) + (lane & 1)) / stream_ctas(p));   // lane 0: begin, lane 1: end
  int cut = x;
  if (x < s.total) {
    stream_locate(p, s, x);
    const int n = stream_item_tiles(p, s);
    if (x - s.g0 <= kStreamSnap) cut = s.g0;
    else if (s.g0 + n - x <= kStreamSnap) cut = s.g0 + n;
  }
  s.pos = __shfl_sync(0xffffffffu, cut, 0); s.end = __shfl_sync(0xffffffffu, cut, 1);
  s.seq = __shfl_sync(0xffffffffu, s.seq, 0); s.chunk = __shfl_sync(0xffffffffu, s.chunk, 0);
  s.i = __shfl_sync(0xffffffffu, s.i, 0); s.g0 = __shfl_sync(0xffffffffu, s.g0, 0);
  s.cached_tiles = __shfl_sync(0xffffffffu, s.cached_tiles, 0); s.final_rows = __shfl_sync(0xffffffffu, s.final_rows, 0);
  s.n_items = __shfl_sync(0xffffffffu, s.n_items, 0); s.item0 = __shfl_sync(0xffffffffu, s.item0, 0);
}
// The next piece of the run.
__device__ __forceinline__ WorkEntry stream_next(const AttnParams &p, StreamState &s) {
  WorkEntry e = {-1, 0, 0, 0, -1, 0};
  if (s.pos >= s.end) return e;
  int n = stream_item_tiles(p, s);
  while (s.pos >= s.g0 + n) {
    s.g0 += n;
    s.i += 2;
    if (s.i >= s.n_items) {
      if (++s.chunk == p.n_chunks) {
        s.chunk = 0;
        do { ++s.seq; stream_sequence(p, s); } while (stream_of(p) >= s.n_items && s.seq + 1 < p.seg.batch);
      }
      s.i = stream_of(p);
    }
    n = stream_item_tiles(p, s);
  }
  e.pair = s.item0 + s.i; e.chunk = s.chunk;
  e.tile0 = s.pos - s.g0;
  e.n_tiles = min(s.end, s.g0 + n) - s.pos;
  s.pos += e.n_tiles;
  // the CTAs that share the item: the last one whose run begins at or before its first tile .. the last one whose run
  // begins inside it (cuts near the edges moved as above)
  const int g = stream_ctas(p);
  auto last_cut_up_to = [&](int x) { return min(g - 1, (int)((((long long)x + 1) * g - 1) / s.total)); };
  const int j0 = last_cut_up_to(s.g0 + min(kStreamSnap, n - 1));
  const int j1 = max(j0, last_cut_up_to(s.g0 + n - kStreamSnap - 1));
  if (j1 > j0) {
    e.split = stream_cta(p) - j0;
    e.fill = stream_cta(p) == j1 ? e.split + 1 : p.n_splits;
    if (e.split < 0 || j1 - j0 >= p.n_splits) { ba_record_status(p.status, BA_ERR_SHAPE); e.pair = -1; }
  }
  return e;
}

// The last own key tile of an item covers the diagonal of the causal range.  When every row of the item
// ends in the tile's first 64 keys (true for every other item: items are 64-token aligned, key tiles 128),
// its second half is masked for all of them: the products and the exponentials of that half are skipped.
__device__ __forceinline__ bool last_tile_is_half(const Work &wk) {
  const Item &it = wk.it;
  if (wk.tile0 + wk.n_tiles != it.n_tiles || it.n_tiles == it.n_cache_tiles) return false;   // the entry does not end the item
  const int last_key0 = it.own_row0 + (it.n_tiles - it.n_cache_tiles - 1) * kBlockN;
  return it.q_row0 + it.q_rows - 1 - last_key0 < kBlockN / 2;
}

// Block-by-block walk of the cached keys: index (cache order) of the block that holds key tile
// `target` (counted over the whole batch).
__device__ __forceinline__ int find_cache_block(const AttnParams &p, int target) { return __ldg(p.seg.cache_tile_block + target); }

// Counter-rotation of query rows [row_begin, row_end) of one tile (fused warm path): dst = R(-delta) src,
// with cs = (cos, sin)(delta * theta_m) of the current cached block.  Both tiles are in the 128-byte
// swizzled layout the tensor maps produce: 64-column regions of 128 rows x 128 bytes, the 16-byte
// chunk c of row r stored at chunk position c ^ (r & 7).  Called by one full warp; a lane keeps its
// chunk column, so its (cos, sin) values are loaded once per block.
__device__ __forceinline__ uint32_t rot_word_adjacent(uint32_t w, float2 cs) {
  const float x = __uint_as_float(w << 16), y = __uint_as_float(w & 0xffff0000u);
  __nv_bfloat162 v = __floats2bfloat162_rn(fmaf(x, cs.x, y * cs.y), fmaf(y, cs.x, -x * cs.y));
  return *reinterpret_cast<uint32_t *>(&v);
}
__device__ __forceinline__ void rot_words_half(uint32_t &a, uint32_t &b, float2 cs0, float2 cs1) {
  // a holds x of pairs m, m+1; b holds their partners y
  const float x0 = __uint_as_float(a << 16), x1 = __uint_as_float(a & 0xffff0000u);
  const float y0 = __uint_as_float(b << 16), y1 = __uint_as_float(b & 0xffff0000u);
  __nv_bfloat162 va = __floats2bfloat162_rn(fmaf(x0, cs0.x, y0 * cs0.y), fmaf(x1, cs1.x, y1 * cs1.y));
  __nv_bfloat162 vb = __floats2bfloat162_rn(fmaf(y0, cs0.x, -x0 * cs0.y), fmaf(y1, cs1.x, -x1 * cs1.y));
  a = *reinterpret_cast<uint32_t *>(&va);
  b = *reinterpret_cast<uint32_t *>(&vb);
}
// One thread rotates one row of a query tile (row r = TMEM lane r = the row whose softmax the
// thread computes).  The (cos, sin) values of the block are the same for every row: `cs` points
// to a copy of them in shared memory, read as warp-wide broadcasts.  The row is loaded in full
// before the arithmetic starts, so that the shared-memory latency is paid once.
template <int D>
__device__ __forceinline__ void rotate_q_row(const uint8_t *__restrict__ src, uint8_t *__restrict__ dst,
                                             const float2 *__restrict__ cs, int layout, int r) {
  constexpr int kRegion = 128 * 128;
  constexpr int kVec = D / 8;                      // 16-byte chunks per row
  const int rb = r * 128, sw = r & 7;
  uint4 v[kVec];
  int off[kVec];
#pragma unroll
  for (int i = 0; i < kVec; ++i) {
    off[i] = (i >> 3) * kRegion + rb + (((i & 7) ^ sw) << 4);     // chunk i of the row: columns 8 i .. 8 i + 7
    v[i] = *reinterpret_cast<const uint4 *>(src + off[i]);
  }
  if (layout == BA_ROPE_ADJACENT) {
#pragma unroll
    for (int i = 0; i < kVec; ++i) {
      const float4 c01 = *reinterpret_cast<const float4 *>(cs + i * 4);
      const float4 c23 = *reinterpret_cast<const float4 *>(cs + i * 4 + 2);
      v[i].x = rot_word_adjacent(v[i].x, make_float2(c01.x, c01.y)); v[i].y = rot_word_adjacent(v[i].y, make_float2(c01.z, c01.w));
      v[i].z = rot_word_adjacent(v[i].z, make_float2(c23.x, c23.y)); v[i].w = rot_word_adjacent(v[i].w, make_float2(c23.z, c23.w));
    }
  } else {
    // pairs (m, m + D/2): chunk i (< kVec / 2) holds x of pairs 8 i .. 8 i + 7, chunk i + kVec / 2 their partners
#pragma unroll
    for (int i = 0; i < kVec / 2; ++i) {
      const float4 *cp = reinterpret_cast<const float4 *>(cs + i * 8);
      const float4 c01 = cp[0], c23 = cp[1], c45 = cp[2], c67 = cp[3];
      uint4 &a = v[i], &b = v[i + kVec / 2];
      rot_words_half(a.x, b.x, make_float2(c01.x, c01.y), make_float2(c01.z, c01.w));
      rot_words_half(a.y, b.y, make_float2(c23.x, c23.y), make_float2(c23.z, c23.w));
      rot_words_half(a.z, b.z, make_float2(c45.x, c45.y), make_float2(c45.z, c45.w));
      rot_words_half(a.w, b.w, make_float2(c67.x, c67.y), make_float2(c67.z, c67.w));
    }
  }
#pragma unroll
  for (int i = 0; i < kVec; ++i) *reinterpret_cast<uint4 *>(dst + off[i]) = v[i];
}

// Cluster launch: the rows of an item are shared out among the CTAs of the cluster (a warp takes whole rows), each row is the
// sum of every CTA's normalised row, weighted by its denominator -- the arithmetic of ba_combine_splits_kernel, through
// distributed shared memory.  rows: fp32 [128][D] of this CTA for query tile 0 (at rows0) and 1 (rows1), 16-byte chunk c of row
// r at chunk position c ^ (r & 7); lse: [2][128].
template <int D>
__device__ __forceinline__ void cluster_merge_rows(const AttnParams &p, const WorkEntry &e, int warp, uint32_t rows0, uint32_t rows1,
                                                   uint32_t lse) {
  constexpr int kLanes = D / 4, kRows = 32 / kLanes;      // lanes per row, rows a warp takes at a time
  const int lane = threadIdx.x & 31, c = lane % kLanes;
  const int n = p.cluster, rank = (int)cluster_rank();
  Item it;
  load_item(p, e.pair, it);
  narrow_item(p, e.fill, it);
  const int q_end = min(it.q_row0 + it.q_rows, p.n_q_rows);
  for (int rr = (rank * 8 + warp) * kRows + lane / kLanes; rr < it.n_qt * 128; rr += n * 8 * kRows) {
    const int t = rr >> 7, r = rr & 127;
    const int tk = it.q_row0 + t * p.tok + (r >> p.hpt_log2), head = e.chunk * p.hpt + (r & (p.hpt - 1));
    if (tk >= q_end) continue;
    const uint32_t at = (t ? rows1 : rows0) + r * (D * 4) + ((c ^ (r & 7)) << 4);
    float ls[kMaxCluster], mx = -INFINITY, den = 0.f;
    float4 x[kMaxCluster], acc = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int s = 0; s < kMaxCluster; ++s) {
      ls[s] = -INFINITY;
      if (s < n) {
        ls[s] = cluster_ld_f32(cluster_map(lse + rr * 4, s));
        x[s] = cluster_ld_v4(cluster_map(at, s));
      }
    }
#pragma unroll
    for (int s = 0; s < kMaxCluster; ++s) mx = fmaxf(mx, ls[s]);
#pragma unroll
    for (int s = 0; s < kMaxCluster; ++s) {
      if (ls[s] == -INFINITY) continue;                   // that CTA saw no key: it holds no row at all
      const float w = __expf(ls[s] - mx);
      den += w;
      acc.x = fmaf(w, x[s].x, acc.x); acc.y = fmaf(w, x[s].y, acc.y); acc.z = fmaf(w, x[s].z, acc.z); acc.w = fmaf(w, x[s].w, acc.w);
    }
    const float inv = 1.f / den;
    acc.x *= inv; acc.y *= inv; acc.z *= inv; acc.w *= inv;
    const size_t row = (size_t)tk * p.Hq + head;
    if (p.out_f32) {
      reinterpret_cast<float4 *>(reinterpret_cast<float *>(p.o) + row * D)[c] = acc;
    } else {
      __nv_bfloat162 a = __floats2bfloat162_rn(acc.x, acc.y), b = __floats2bfloat162_rn(acc.z, acc.w);
      uint2 w2 = make_uint2(*reinterpret_cast<uint32_t *>(&a), *reinterpret_cast<uint32_t *>(&b));
      reinterpret_cast<uint2 *>(reinterpret_cast<__nv_bfloat16 *>(p.o) + row * D)[c] = w2;
    }
    if (p.lse && c == 0) p.lse[row] = mx + logf(den);
  }
}

template <int D, int kVariant>
__global__ void __launch_bounds__(kThreads, 1)
ba_attend_sm100_kernel(const __grid_constant__ CUtensorMap tmap_q, const __grid_constant__ CUtensorMap tmap_k,
                       const __grid_constant__ CUtensorMap tmap_v, const __grid_constant__ CUtensorMap tmap_kc,
                       const __grid_constant__ CUtensorMap tmap_vc, const __grid_constant__ CUtensorMap tmap_o, const AttnParams p) {
  using L = Layout<D>;
  constexpr bool kFused = is_fused(kVariant), kDeep = is_deep(kVariant);
  // Half tiles at the ends of cached blocks, values walked in a pool: 16 requests over 20 blocks of 50-500 tokens 1401 -> 1377 us
  // (four layers).  Not on the fused path: the flags cost its product thread more than the halves save.
  constexpr bool kWalks = kDeep;
  constexpr bool kClustered = kVariant == kFusedCluster || kVariant == kDeepCluster || kVariant == kSharedCluster;
  constexpr bool kSolo = kVariant == kSharedCluster;
  constexpr bool kReady = kVariant == kPlain || kVariant == kDeepRing;
  // The rescaling of O stays a loop (kFusedCluster, eight requests of 12 cached blocks of 37-611 and 32 final tokens: 262 -> 255 us),
  // but not in kFusedPath: with one query tile nothing else runs meanwhile, and the loop takes longer (32 x 1000 cached tokens and
  // 1 / 32 final ones, eight layers, as a loop and unrolled: 439 and 421, 452 and 439 us; two query tiles: 519 and 521).
  constexpr int kRescaleUnroll = kVariant == kFusedPath ? D / 32 : 1;
  // (layouts a variant is never launched with are not in its code: a short launch pays for every instruction it passes; a 32-layer
  // prompt of 2500 cached tokens 824 -> 795 us)
  const int balanced = kClustered || kDeep ? 0 : p.balanced, stream = kClustered ? 0 : p.stream, persistent = kClustered ? 0 : p.persistent;
  constexpr int kStages = kDeep ? 4 : 3;
  // setmaxnreg is a warpgroup-wide instruction: the four service warps (8-11) must ask for the same count
  constexpr int kServiceRegs = kFused ? kServiceRegsFused : kServiceRegsPlain;
  constexpr int kSoftmaxRegs = kFused ? kSoftmaxRegsFused : kSoftmaxRegsPlain;
  constexpr int kProdRegs = kServiceRegs, kMmaRegs = kServiceRegs, kSpareRegs = kServiceRegs;
  extern __shared__ uint8_t smem_raw[];
  uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  Ctrl *ctrl = reinterpret_cast<Ctrl *>(smem + L::kCtrl);

  const int tid = threadIdx.x, warp = tid >> 5;

  if (tid == 0) {
    for (int b = 0; b < 2; ++b)
      for (int t = 0; t < 2; ++t) { mbar_init(&ctrl->q_full[b][t], 1); mbar_init(&ctrl->q_empty[b][t], kDeep ? 1 : 4); }
    for (int s = 0; s < kStages; ++s) { mbar_init(&ctrl->kv_full[s], 1); mbar_init(&ctrl->kv_empty[s], 1); }
    for (int t = 0; t < 2; ++t) {
      mbar_init(&ctrl->s_full[t], 1); mbar_init(&ctrl->p_full[t][0], 128); mbar_init(&ctrl->p_full[t][1], 128);
      mbar_init(&ctrl->o_done[t], 1); mbar_init(&ctrl->o_free[t], 128); mbar_init(&ctrl->out_staged[t], 128);
      mbar_init(&ctrl->qr_full[t][0], 4); mbar_init(&ctrl->qr_full[t][1], 4); mbar_init(&ctrl->cs_full[t], D / 2);
      mbar_init(&ctrl->qraw_full[t], 1);
    }
    mbar_init(&ctrl->solo_full, 128);
    for (int k = 0; k < kWorkSlots; ++k) { mbar_init(&ctrl->work_full[k], 1); mbar_init(&ctrl->work_empty[k], 9); }
    if (kClustered) ctrl->work_ring[0].pair = -1;
    ctrl->abort_flag = 0; ctrl->n_staged_out[0] = 0; ctrl->n_staged_out[1] = 0;
    fence_barrier_init();
  }
  if (warp == 9) { tmem_alloc(&ctrl->tmem_base, 512); tmem_relinquish(); }
  if (warp == 10 && elect_one()) {
    prefetch_tmap(&tmap_q); prefetch_tmap(&tmap_k); prefetch_tmap(&tmap_v); prefetch_tmap(&tmap_kc); prefetch_tmap(&tmap_vc);
  }
  ba_pdl_wait();
  // The CTA's first entry is known from its index: the scheduling warp looks it up while the others set the CTA up.
  // Inconsistent tables: no attention work is taken, a background job still runs.
  int n_items = 0;
  WorkEntry first = {-1, 0, 0, 0, -1, 0};
  if (warp == 8) {
    const bool fit = kVariant != kPlain || partials_fit(p.seg.totals, p.final_only, p.n_splits, p.n_part_rows);
    n_items = count_items(p);
    if (!fit && n_items > 0) {
      ba_record_status(p.status, BA_ERR_SHAPE);            // the tables describe another launch than the host sized
      n_items = 0;
    }
    if (kClustered) first = cluster_entry(p, n_items);
    else if (!balanced && !stream) first = list_entry(p, n_items, (int)blockIdx.x);
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = ctrl->tmem_base;
  volatile int *abort_flag = &ctrl->abort_flag;
  ReadyItem *ready = reinterpret_cast<ReadyItem *>(smem + L::kCtrl + kReadyOff);
  ba_pdl_trigger();

  // The CTA is persistent: its producer thread draws entries of the global work list from an
  // atomic counter (heaviest items first, whichever SM is free takes the next) and publishes them
  // to the other roles through a small ring; mbarrier phases simply keep counting across items, so the producer and the MMA warp run ahead into the next item while
  // the softmax warps still write out the previous one.
  // The softmax warps keep a whole 128-column row in registers; the service warps (8-11) need few.
  if (warp == 8) {
    // ------------------------------------------------------------ TMA producer
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kProdRegs));
    // balanced launch, a CTA that shares the front key tiles: prefix sum of the front tiles of every item (the
    // same for every head chunk), one item per lane, kept in shared memory for the scheduling thread
    int *bal_cu = reinterpret_cast<int *>(smem + L::kCtrl + kBalTableOff);
    int bal_np = 0;
    if (balanced && n_items > 0) {
      bal_np = n_items;
      if (bal_np < 1 || bal_np > kBalMaxPairs || bal_np * p.n_chunks != balanced) {
        ba_record_status(p.status, BA_ERR_SHAPE);          // the tables describe another launch than the host sized
        bal_np = 0;
      } else if ((int)blockIdx.x >= balanced) {
        const int lane = tid & 31;
        int carry = 0;
        for (int base = 0; base < bal_np; base += 32) {
          const int i = base + lane;
          int x = 0;
          if (i < bal_np) {
            Item it;
            load_item(p, bal_np - 1 - i, it);
            x = max(0, it.n_tiles - p.bal_len);
          }
#pragma unroll
          for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
          }
          if (i < bal_np) bal_cu[i + 1] = carry + x;
          carry += __shfl_sync(0xffffffffu, x, 31);
        }
        if (lane == 0) bal_cu[0] = 0;
        __syncwarp();
      }
    }
    StreamState ss = {};
    if (stream && n_items > 0) stream_start(p, ss);
    if (elect_one()) {
      // balanced launch: run [bal_pos, bal_end) of the front tiles of all (chunk, item), bal_hm of them per chunk
      int bal_pos = 0, bal_end = 0, bal_hm = 0, bal_nh = 0;
      long long bal_all = 0;
      if (bal_np > 0 && (int)blockIdx.x >= balanced) {
        bal_hm = bal_cu[bal_np];
        bal_all = (long long)bal_hm * p.n_chunks;
        bal_nh = (int)gridDim.x - balanced;
        const int j = (int)blockIdx.x - balanced;
        bal_pos = (int)(bal_all * j / bal_nh);
        bal_end = (int)(bal_all * (j + 1) / bal_nh);
      }
      auto balanced_entry = [&](int n_done) -> WorkEntry {
        WorkEntry e = {-1, 0, 0, 0, -1, 0};
        if (bal_np == 0) return e;
        const int b = (int)blockIdx.x;
        if (b < balanced) {                              // the last bal_len key tiles of item b
          if (n_done > 0) return e;
          Item it;
          const int pair = bal_np - 1 - b % bal_np;
          load_item(p, pair, it);
          e.pair = pair; e.chunk = b / bal_np;
          e.tile0 = max(0, it.n_tiles - p.bal_len);
          e.n_tiles = it.n_tiles - e.tile0;
          e.split = 0;
          e.fill = e.tile0 == 0 ? 1 : p.n_splits;           // nothing in front: the other slots stay empty
          return e;
        }
        if (bal_pos >= bal_end) return e;
        const int chunk = bal_pos / bal_hm, r = bal_pos - chunk * bal_hm;
        int lo = 0, hi = bal_np + 1;                        // item i with bal_cu[i] <= r < bal_cu[i + 1]
        while (lo < hi) { const int mid = (lo + hi) >> 1; if (bal_cu[mid] <= r) lo = mid + 1; else hi = mid; }
        const int i = lo - 1;
        const int front_end = chunk * bal_hm + bal_cu[i + 1];
        const int n = min(bal_end, front_end) - bal_pos;
        // the slot counts the CTAs from the one that holds the first front tile of the item
        const long long g0 = (long long)chunk * bal_hm + bal_cu[i];
        const int j_first = (int)(((g0 + 1) * bal_nh - 1) / bal_all);
        e.split = 1 + ((int)blockIdx.x - balanced) - j_first;
        if (e.split >= p.n_splits) { ba_record_status(p.status, BA_ERR_SHAPE); return e; }
        e.pair = bal_np - 1 - i; e.chunk = chunk;
        e.tile0 = r - bal_cu[i]; e.n_tiles = n;
        e.fill = bal_pos + n == front_end ? e.split + 1 : p.n_splits;
        bal_pos += n;
        return e;
      };
      int gidx = 0;                       // K/V tiles requested so far (ring position)
      int n_loaded = 0;                   // entries whose queries have been requested so far
      int uses1[2] = {0, 0};              // of those in buffer pair b, the ones with a second query tile
      bool ok = true;
      Work wk;
      int n_work = 0;                    // work entries published so far
      for (;;) {
        // scheduler: take the next entry of the global work list and publish it to the other roles
        const int slot = n_work & (kWorkSlots - 1);
        ok = mbar_wait(&ctrl->work_empty[slot], ((n_work / kWorkSlots) & 1) ^ 1, abort_flag);
        if (!ok) break;
        // balanced launch: the next piece of this CTA's share; persistent launch: next entry of the global list;
        // one-item launch: this CTA's own entry, then stop
        WorkEntry e = {-1, 0, 0, 0, -1, 0};
        if (balanced) e = balanced_entry(n_work);
        else if (stream) e = stream_next(p, ss);
        else if (n_work == 0) e = first;
        else if (persistent) e = list_entry(p, n_items, (int)gridDim.x + atomicAdd(p.counters, 1));
        const bool more = load_work<kClustered>(p, e, wk);
        if (!more) e.pair = -1;
        ctrl->work_ring[slot] = e;
        if (kReady && more)
          ready[slot] = {wk.it.q_row0, wk.it.q_rows, wk.it.own_row0, wk.it.cache_len, wk.it.n_cache_tiles, wk.it.n_tiles, wk.it.ctile0, 0};
        mbar_arrive(&ctrl->work_full[slot]);
        ++n_work;
        if (!more) break;
        if (wk.n_tiles == 0) continue;
        const Item &it = wk.it;
        if (!kFused) {      // (on the fused path the softmax warps fetch the query tiles themselves)
          // a Q buffer is free once the rows of the entry that used it have been written out
          const int qb = p.q_double ? (n_loaded & 1) : 0;            // buffer pair of this entry
          const int q_use = p.q_double ? (n_loaded >> 1) : n_loaded;  // earlier entries that used it
          ok = mbar_wait(&ctrl->q_empty[qb][0], (q_use & 1) ^ 1, abort_flag);
          if (!kDeep && ok && it.n_qt == 2) ok = mbar_wait(&ctrl->q_empty[qb][1], ((qb ? uses1[1] : uses1[0]) & 1) ^ 1, abort_flag);
          if (!ok) break;
          ++n_loaded;
          if (it.n_qt == 2) { if (qb) ++uses1[1]; else ++uses1[0]; }
          for (int t = 0; t < 2; ++t) {
            if (t >= it.n_qt) { mbar_arrive(&ctrl->q_full[qb][t]); continue; }   // (every entry moves both barriers on)
            mbar_arrive_expect_tx(&ctrl->q_full[qb][t], L::kTileBytes);
            uint8_t *dst = smem + (qb ? L::kBg + t * L::kTileBytes : (t ? L::kQ1 : L::kQ0));
            for (int c = 0; c < L::kChunks; ++c)
              tma_load_3d(dst + c * L::kRegionBytes, &tmap_q, &ctrl->q_full[qb][t], c * 64, wk.head0,
                          it.q_row0 + t * p.tok);
          }
        }
        // walk mode: cached keys are taken block by block (block pc, row offset poff inside it).  The
        // current block's length and first rows sit in registers and the next block's are fetched a
        // whole block ahead, so that no tile waits for a table look-up.
        int pc = 0, poff = 0;
        int c_len = 0, k_base = 0, v_base = 0, n_len = 0, n_kbase = 0, n_vbase = 0;
        // (for a paged operand the "base" of a block is the start of its page list)
        auto load_block = [&](int b, int &len, int &kb, int &vb) {
          if (b >= p.seg.n_cached_blocks) return;
          const int c0 = __ldg(p.seg.cache_cu + b);
          len = __ldg(p.seg.cache_cu + b + 1) - c0;
          const int pg = p.page_cu ? __ldg(p.page_cu + b) : 0;
          kb = p.k_paged ? pg : (p.k_src_off ? __ldg(p.k_src_off + b) : c0);
          vb = p.v_paged ? pg : (p.v_src_off ? __ldg(p.v_src_off + b) : c0);
        };
        if (p.walk && wk.tile0 < it.n_cache_tiles) {
          const int target = it.ctile0 + wk.tile0;
          pc = find_cache_block(p, target);
          poff = (target - __ldg(p.seg.cache_tile_cu + pc)) * kBlockN;
          load_block(pc, c_len, k_base, v_base);
          load_block(pc + 1, n_len, n_kbase, n_vbase);
        }
        // one 128-row tile of a paged operand: a box per page (pages of 128 rows or more hold whole tiles).
        // Parts of the tile past the end of the block are fetched from the block's last page: they are
        // masked, but what the tensor core multiplies by zero must still be finite.
        auto load_paged_tile = [&](uint8_t *dst, const CUtensorMap *m, uint64_t *bar, int list0, int off, int len) {
          const int page_rows = 1 << p.page_lg;
          const int sub_rows = min(kBlockN, page_rows), n_sub = kBlockN / sub_rows;
          const int last_page = (len - 1) >> p.page_lg;
          for (int sb = 0; sb < n_sub; ++sb) {
            const int t0 = off + sb * sub_rows;
            const int page = min(t0 >> p.page_lg, last_page);
            const int row = (__ldg(p.page_idx + list0 + page) << p.page_lg) + (t0 & (page_rows - 1));
            for (int c = 0; c < L::kChunks; ++c)
              tma_load_3d(dst + c * L::kRegionBytes + sb * sub_rows * 128, m, bar, c * 64, wk.kv_head, row);
          }
        };
        // (one loop for both orders, with a tile's rows kept for its values, cost the kernels that have one order 1-2 %: cold prompt of
        // 7200 tokens 783 -> 798 us)
        if constexpr (!kSolo) {
          for (int j = 0; j < wk.n_tiles && ok; ++j) {
            const int jt = wk.tile0 + j;
            const bool cached = jt < it.n_cache_tiles;
            int k_row, v_row, t_off = 0, t_len = 0, t_kbase = 0, t_vbase = 0;
            bool k_pg = false, v_pg = false;
            if (!cached) {
              k_row = v_row = it.own_row0 + (jt - it.n_cache_tiles) * kBlockN;
            } else if (!p.walk) {
              k_row = v_row = it.cache_row0 + jt * kBlockN;
            } else {
              k_row = k_base + poff;
              v_row = v_base + poff;
              k_pg = p.k_paged; v_pg = p.v_paged;
              t_off = poff; t_len = c_len; t_kbase = k_base; t_vbase = v_base;
              ctrl->tile_valid[(gidx >> 1) & 7] = min(kBlockN, c_len - poff);   // read by the softmax warps
              poff += kBlockN;
              if (poff >= c_len) {
                ++pc; poff = 0;
                c_len = n_len; k_base = n_kbase; v_base = n_vbase;
                load_block(pc + 1, n_len, n_kbase, n_vbase);
              }
            }
            for (int kv = 0; kv < 2; ++kv) {
              const int stage = gidx % kStages;
              ok = mbar_wait(&ctrl->kv_empty[stage], ((gidx / kStages) & 1) ^ 1, abort_flag);
              if (!ok) break;
              const CUtensorMap *m = cached ? (kv ? &tmap_vc : &tmap_kc) : (kv ? &tmap_v : &tmap_k);
              uint8_t *dst = smem + L::kRing + stage * L::kTileBytes;
              mbar_arrive_expect_tx(&ctrl->kv_full[stage], L::kTileBytes);
              if (kv ? v_pg : k_pg) {
                load_paged_tile(dst, m, &ctrl->kv_full[stage], kv ? t_vbase : t_kbase, t_off, t_len);
              } else {
                for (int c = 0; c < L::kChunks; ++c)
                  tma_load_3d(dst + c * L::kRegionBytes, m, &ctrl->kv_full[stage], c * 64, wk.kv_head, kv ? v_row : k_row);
              }
              ++gidx;
            }
          }
        } else {
          // one tile of K (kv = 0) or V into the next stage of the ring
          struct TileRows { int k_row, v_row, off, len, kbase, vbase; bool cached, k_pg, v_pg; };
          auto load_tile = [&](const TileRows &x, int kv) {
            const int stage = gidx % kStages;
            ok = mbar_wait(&ctrl->kv_empty[stage], ((gidx / kStages) & 1) ^ 1, abort_flag);
            if (!ok) return;
            const CUtensorMap *m = x.cached ? (kv ? &tmap_vc : &tmap_kc) : (kv ? &tmap_v : &tmap_k);
            uint8_t *dst = smem + L::kRing + stage * L::kTileBytes;
            mbar_arrive_expect_tx(&ctrl->kv_full[stage], L::kTileBytes);
            if (kv ? x.v_pg : x.k_pg) {
              load_paged_tile(dst, m, &ctrl->kv_full[stage], kv ? x.vbase : x.kbase, x.off, x.len);
            } else {
              for (int c = 0; c < L::kChunks; ++c)
                tma_load_3d(dst + c * L::kRegionBytes, m, &ctrl->kv_full[stage], c * 64, wk.kv_head, kv ? x.v_row : x.k_row);
            }
            ++gidx;
          };
          const bool solo = is_solo<kSolo>(wk);
          const int first_tile = gidx >> 1;   // tiles of all earlier entries (the other roles count the same way)
          TileRows x = {}, before = {};
          for (int j = 0; j < wk.n_tiles + (solo ? 1 : 0) && ok; ++j) {
            if (j < wk.n_tiles) {
              const int jt = wk.tile0 + j;
              x = {};
              x.cached = jt < it.n_cache_tiles;
              if (!x.cached) {
                x.k_row = x.v_row = it.own_row0 + (jt - it.n_cache_tiles) * kBlockN;
              } else if (!p.walk) {
                x.k_row = x.v_row = it.cache_row0 + jt * kBlockN;
              } else {
                x.k_row = k_base + poff;
                x.v_row = v_base + poff;
                x.k_pg = p.k_paged; x.v_pg = p.v_paged;
                x.off = poff; x.len = c_len; x.kbase = k_base; x.vbase = v_base;
                ctrl->tile_valid[(first_tile + j) & 7] = min(kBlockN, c_len - poff);   // read by the softmax warps
                poff += kBlockN;
                if (poff >= c_len) {
                  ++pc; poff = 0;
                  c_len = n_len; k_base = n_kbase; v_base = n_vbase;
                  load_block(pc + 1, n_len, n_kbase, n_vbase);
                }
              }
              load_tile(x, 0);
            }
            if (!ok) break;
            if (!solo) {
              load_tile(x, 1);
            } else {
              if (j > 0) load_tile(before, 1);
              before = x;
            }
          }
        }
        if (kClustered) break;
      }
      if (!ok) {
        // leave no copy in flight: wait (bounded) for the tiles already requested
        for (int idx = max(0, gidx - kStages); idx < gidx; ++idx)
          for (uint32_t spin = 0; spin < (1u << 20); ++spin)
            if (mbar_try_wait(&ctrl->kv_full[idx % kStages], (idx / kStages) & 1)) break;
      }
    }
    if (kClustered) { __syncwarp(); cluster_sync(); }      // (the softmax warps merge between this one and the next)
  } else if (warp == 9) {
    // ------------------------------------------------------------ MMA issuer
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kMmaRegs));
    if (elect_one()) {
      const uint32_t tS[2] = {tmem, tmem + 128};
      const uint32_t tO[2] = {tmem + 256, tmem + 384};
      constexpr uint32_t idesc_qk = make_idesc_bf16(128, kBlockN, 0);
      constexpr uint32_t idesc_qk_half = make_idesc_bf16(128, kBlockN / 2, 0);   // keys 0..63 of the tile only
      constexpr uint32_t idesc_pv = make_idesc_bf16(128, D, 1);
      const uint32_t q_addr[2] = {smem_u32(smem + L::kQ0), smem_u32(smem + L::kQ1)};
      const uint32_t ring = smem_u32(smem + L::kRing);
      bool ok = true;
      auto wait_kv = [&](int idx) { return mbar_wait(&ctrl->kv_full[idx % kStages], (idx / kStages) & 1, abort_flag); };
      // descriptors differ only in their start-address field: build them once, add offsets (>> 4)
      const uint64_t q_desc[2] = {make_smem_desc(q_addr[0], 16, 1024), make_smem_desc(q_addr[1], 16, 1024)};
      const uint64_t k_desc0 = make_smem_desc(ring, 16, 1024);
      const uint64_t v_desc0 = make_smem_desc(ring, L::kRegionBytes, 1024);
      Work wk = {};
      bool half_last = false;              // the entry's last key tile is used in its first 64 keys only
      int entry_tiles = 0;
      // a cached tile whose block ends in its first 64 keys (walk mode; the producer's word comes with the tile)
      int first_tile = 0;                  // tiles of all earlier entries
      auto cached_half = [&](int jrel) -> bool {
        return kWalks && p.walk && wk.tile0 + jrel < wk.it.n_cache_tiles && ctrl->tile_valid[(first_tile + jrel) & 7] <= kBlockN / 2;
      };
      auto issue_qk_with = [&](int t, int jrel, int idx, uint64_t qd) {
        const uint64_t kd = k_desc0 + (uint64_t)(((idx % kStages) * L::kTileBytes) >> 4);
        const uint32_t idesc = ((half_last && jrel + 1 == entry_tiles) || cached_half(jrel)) ? idesc_qk_half : idesc_qk;
#pragma unroll
        for (int k = 0; k < D / 16; ++k) {
          const uint64_t off = (uint64_t)(((k >> 2) * L::kRegionBytes + (k & 3) * 32) >> 4);
          mma_ss(tS[t], qd + off, kd + off, idesc, k > 0);
        }
        mma_commit(&ctrl->s_full[t]);
      };
      // half = 0: keys 0..63 of the tile, half = 1: keys 64..127
      auto issue_pv = [&](int t, int idx, bool first, int half) {
        const uint64_t vd = v_desc0 + (uint64_t)(((idx % kStages) * L::kTileBytes) >> 4);
#pragma unroll
        for (int k = half * 4; k < half * 4 + 4; ++k)
          mma_ts(tO[t], tS[t] + k * 8, vd + (uint64_t)((k * 2048) >> 4), idesc_pv, (!first || k > 0) ? 1u : 0u);
      };
      int gidx = 0;                        // K/V tiles consumed so far (ring position)
      int q_uses[2] = {0, 0};              // items in which query tile t was loaded
      int p_uses[2] = {0, 0};              // P tiles of query tile t consumed
      int n_work = 0;
      // Every loop over the query tile t below is unrolled, so that t is a constant and the small
      // per-tile arrays live in registers: this thread's issue latency is on the critical path.
      // fused path: a "version" of query tile t is the tile prepared for one key range of the entry --
      // rotated for one cached block, or plain for the final block's own keys.  The softmax threads
      // prepare versions in order into alternating buffers; both sides count them alike.
      const uint64_t qb_desc[2] = {make_smem_desc(smem_u32(smem + L::kBg), 16, 1024),         // second buffers
                                   make_smem_desc(smem_u32(smem + L::kBg + L::kTileBytes), 16, 1024)};
      int n_ver[2] = {0, 0};               // versions of query tile t taken so far
      int ver_end[2] = {-1, -1};           // the current version of tile t serves cached key tiles below this index
      int walk_pc = 0, walk_end = -1;      // block of the current cached tile and the tile index where it ends
      int cached_end = 0;                  // tiles [tile0, cached_end) of the entry are cached keys
      int q_buf = 0;                       // plain path: buffer pair that holds the entry's query tiles
      bool solo = false;                   // one query tile, key tiles shared by the softmax groups (is_solo)
      // S_t = Q_t K^T for tile `jrel` of the entry, whose keys sit at ring position idx
      auto issue_qk = [&](int t, int jrel, int idx) -> bool {
        if (!kFused) { const int q = solo ? 0 : t; issue_qk_with(t, jrel, idx, q_buf ? qb_desc[q] : q_desc[q]); return true; }
        const int jt = wk.tile0 + jrel;
        bool change = false;
        if (jt < cached_end) {
          const int g = wk.it.ctile0 + jt;
          if (g >= ver_end[t]) {                           // first key tile of another cached block
            if (walk_end < 0) { walk_pc = find_cache_block(p, g); walk_end = __ldg(p.seg.cache_tile_cu + walk_pc + 1); }
            while (g >= walk_end) { ++walk_pc; walk_end = __ldg(p.seg.cache_tile_cu + walk_pc + 1); }
            ver_end[t] = walk_end;
            change = true;
          }
        } else if (ver_end[t] != 0x7fffffff) {             // first of the final block's own key tiles
          ver_end[t] = 0x7fffffff;
          change = true;
        }
        if (change) {
          BA_TR(5, n_ver[t] & 63, t * 2);
          if (!mbar_wait(&ctrl->qr_full[t][n_ver[t] & 1], (n_ver[t] >> 1) & 1, abort_flag)) return false;
          BA_TR(5, n_ver[t] & 63, t * 2 + 1);
          ++n_ver[t];
          tc_fence_after();
        }
        issue_qk_with(t, jrel, idx, ((n_ver[t] - 1) & 1) ? qb_desc[t] : q_desc[t]);
        return true;
      };
      for (;;) {
        const int slot = n_work & (kWorkSlots - 1);
        ok = mbar_wait(&ctrl->work_full[slot], (n_work / kWorkSlots) & 1, abort_flag);
        if (!ok) break;
        const WorkEntry e = ctrl->work_ring[slot];
        ++n_work;
        if (!(kReady ? ready_work(p, e, ready[slot], wk) : load_work<kClustered>(p, e, wk))) break;
        mbar_arrive(&ctrl->work_empty[slot]);          // the entry has been decoded into registers
        const int n_tiles = wk.n_tiles, n_qt = wk.it.n_qt;
        if (n_tiles == 0) continue;
        half_last = last_tile_is_half(wk);
        entry_tiles = n_tiles;
        first_tile = gidx >> 1;
        solo = is_solo<kSolo>(wk);
        walk_end = -1; ver_end[0] = ver_end[1] = -1;
        cached_end = min(wk.tile0 + n_tiles, wk.it.n_cache_tiles);
        if (!kFused) {
          // (query tile 0 is part of every entry: q_uses[0] counts the entries)
          q_buf = p.q_double ? (q_uses[0] & 1) : 0;
          const int q_use = p.q_double ? (q_uses[0] >> 1) : q_uses[0];
#pragma unroll
          for (int t = 0; t < 2; ++t)
            if (t < n_qt && ok) ok = mbar_wait(&ctrl->q_full[q_buf][t], q_use & 1, abort_flag);
        }
        if (ok) ok = wait_kv(gidx);
        if (!ok) break;
        tc_fence_after();
#pragma unroll
        for (int t = 0; t < 2; ++t)
          if (t < n_qt && ok) ok = issue_qk(t, 0, gidx);
        if (!ok) break;
        mma_commit(&ctrl->kv_empty[gidx % kStages]);
        if (solo) {
          ok = wait_kv(gidx + 1);
          if (!ok) break;
          tc_fence_after();
          issue_qk(1, 1, gidx + 1);
          mma_commit(&ctrl->kv_empty[(gidx + 1) % kStages]);
        }
        if (kDeep && n_tiles <= (solo ? 2 : 1)) mma_commit(&ctrl->q_empty[0][0]);
        // Round i: tile i for every query tile, or (solo) tiles 2 i and 2 i + 1.
        for (int i = 0; solo ? 2 * i < n_tiles : i < n_tiles; ++i) {
          int iv = gidx + 2 * i + 1, ik = gidx + 2 * i + 2;         // ring positions of V_j and of K of the tile S_t takes next
          BA_TR(3, i, 0);
          if (!solo) ok = wait_kv(iv);
          BA_TR(3, i, 1);
#pragma unroll
          for (int t = 0; t < 2; ++t) {
            const int j = solo ? 2 * i + t : i, jn = j + (solo ? 2 : 1);
            if (!ok || (solo ? j >= n_tiles : t >= n_qt)) continue;
            const bool last = jn >= n_tiles;
            if (solo) {                                    // K_0, K_1, V_0, K_2, V_1, .., K_(n-1), V_(n-2), V_(n-1)
              iv = gidx + 2 * j + (j + 1 < n_tiles ? 2 : 1);
              ik = gidx + 2 * j + 3;
              ok = wait_kv(iv);
              if (!ok) continue;
            }
            BA_TR(2, i, t * 4 + 0);
            // the first PV of an item overwrites O_t: the previous item's rows must have been read out
            if (i == 0) { ok = mbar_wait(&ctrl->o_free[t], (q_uses[t] & 1) ^ 1, abort_flag); if (!ok) continue; }
            ok = mbar_wait(&ctrl->p_full[t][0], p_uses[t] & 1, abort_flag);
            if (!ok) continue;
            tc_fence_after();
            BA_TR(2, i, t * 4 + 1);
            issue_pv(t, iv, i == 0, 0);
            // the next K is needed right after the second half of PV: make sure of it while P is still
            // being finished, off the critical path
            if ((t == 0 || solo) && !last) { BA_TR(3, i, 2); ok = wait_kv(ik); if (!ok) continue; BA_TR(3, i, 3); }
            ok = mbar_wait(&ctrl->p_full[t][1], p_uses[t] & 1, abort_flag);
            if (!ok) continue;
            tc_fence_after();
            if (!(j + 1 == n_tiles && half_last) && !cached_half(j)) issue_pv(t, iv, i == 0, 1);
            ++p_uses[t];
            BA_TR(2, i, t * 4 + 2);
            if (last) mma_commit(&ctrl->o_done[t]);
            if (solo || t + 1 == n_qt) mma_commit(&ctrl->kv_empty[iv % kStages]);
            if (!last) {
              ok = issue_qk(t, jn, ik);
              if (!ok) continue;
              BA_TR(2, i, t * 4 + 3);
              if (solo || t + 1 == n_qt) {
                mma_commit(&ctrl->kv_empty[ik % kStages]);
                if (kDeep && jn + 1 == n_tiles) mma_commit(&ctrl->q_empty[0][0]);   // that was the entry's last QK^T
              }
            }
          }
          if (!ok) break;
        }
        if (!ok) break;
        gidx += 2 * n_tiles;
#pragma unroll
        for (int t = 0; t < 2; ++t)
          if (t < n_qt || solo) ++q_uses[t];
        if (kClustered) break;                             // (one entry)
      }
    }
    if (kClustered) { __syncwarp(); cluster_sync(); }
  } else if (warp >= 10) {
    // ------------------------------------------------------------ spare warps: background re-encoding
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kSpareRegs));
    if (p.bg.n_rows > 0) {
      // each spare warp runs the staged engine with its own two 16 KB stages; chunks are drawn from a
      // device-wide counter, so the job spreads over every CTA of the launch, early and late ones
      const int bw = warp - 10;
      ba_bg_smem *bsm = reinterpret_cast<ba_bg_smem *>(smem + L::kCtrl + 1024) + bw;
      if ((tid & 31) == 0) { mbar_init(&bsm->bar[0], 1); mbar_init(&bsm->bar[1], 1); fence_barrier_init(); }
      __syncwarp();
      ba_reencode_background(p.bg, p.counters + 1, smem + L::kBg + bw * 2 * kBgStageBytes, bsm, p.bg_rows_per_chunk,
                             p.status, [&](uint64_t *bar, uint32_t parity) { return mbar_wait(bar, parity, abort_flag); });
    }
    if (kClustered) { __syncwarp(); cluster_sync(); }
  } else {
    // ------------------------------------------------------------ softmax, one thread per tile row
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kSoftmaxRegs));
    const int t = warp >> 2;
    const int r = tid & 127;
    const uint32_t lane_off = (uint32_t)((warp & 3) * 32) << 16;
    const uint32_t tS = tmem + t * 128 + lane_off;
    const uint32_t tO = tmem + 256 + t * 128 + lane_off;
    const float sl = p.scale_log2;
    int s_uses = 0;                       // S tiles of this query tile consumed so far
    int o_uses = 0;                       // entries that used this group's accumulator so far
    int n_staged = 0;                     // fused: (cos, sin) rows staged so far by this group
    int n_made = 0;                       // fused: versions of this query tile prepared so far
    int tiles_before = 0;                 // key tiles of all earlier items (the producer counts the same way)
    int n_loaded = 0;                     // entries with key tiles so far (the producer counts the same way)
    int out_pending = -1;                 // query buffer pair the copy engine may still be reading (thread 0 of the group)
    auto release_out = [&]() {
      if (kVariant == kPlain && out_pending >= 0) {
        bulk_wait_read();
        mbar_arrive_n(&ctrl->q_empty[out_pending][t], 4);
        out_pending = -1;
      }
      __syncwarp();
    };
    bool ok = true;
    Work wk;
    int n_work = 0;
    for (;;) {
      const int slot = n_work & (kWorkSlots - 1);
      ok = mbar_wait(&ctrl->work_full[slot], (n_work / kWorkSlots) & 1, abort_flag);
      if (!ok) break;
      const WorkEntry e = ctrl->work_ring[slot];
      ++n_work;
      if (!(kReady ? ready_work(p, e, ready[slot], wk) : load_work<kClustered>(p, e, wk))) break;
      __syncwarp();
      if ((tid & 31) == 0) mbar_arrive(&ctrl->work_empty[slot]);   // one arrival per softmax warp
      const Item &it = wk.it;
      const int n_tiles = wk.n_tiles, tile0 = wk.tile0, head0 = wk.head0;
      const bool half_last = last_tile_is_half(wk);
      release_out();
      const bool solo = is_solo<kSolo>(wk);
      const int j0 = solo ? t : 0;         // this group's key tiles: j0, j0 + 1 (solo: j0 + 2), ..
      if (t < it.n_qt || solo) {
      const int tq = solo ? 0 : t;
      // rows past the block behave like its last row
      const int tok_c = min(it.q_row0 + tq * p.tok + (r >> p.hpt_log2), it.q_row0 + it.q_rows - 1);
      float m_used = -INFINITY, l = 0.f;

      // fused path: this thread prepares row r of every version of query tile t (see the MMA warp):
      // the plain tile is fetched by the copy engine into the buffer the version will live in and, for a
      // cached block, every thread rotates its row there in place.  The first version of an entry is made on the spot; every later
      // one is begun after one tile of its predecessor and finished after the next, or at the latest
      // when its first key tile is next.
      const int tile_end = tile0 + n_tiles;
      const int cached_end = min(tile_end, it.n_cache_tiles);          // tiles [tile0, cached_end) are cached keys
      int f_pc = 0;                        // cached block of the version being prepared / in use
      int next_start = tile_end;           // first tile of the next version (tile_end: there is none)
      int prep = 0;                        // next version: 0 not begun, 1 row being fetched, 2 ready
      // The block's (cos, sin) row goes through shared memory: thread r < D/2 of the group holds
      // pair r, fetched one block ahead (cs_next), and the group's 128 threads wait for all of them.
      float2 *cs_stage = reinterpret_cast<float2 *>(smem + L::kCtrl + 1024) + t * 64;
      float2 cs_next = make_float2(1.f, 0.f);
      auto fetch_cs = [&](int pc) {
        if (r < D / 2 && pc < p.seg.n_cached_blocks) cs_next = __ldg(p.q_rope + (size_t)pc * (D / 2) + r);
      };
      auto ver_buf = [&](int v) { return smem + ((v & 1) ? L::kBg : L::kQ0) + t * L::kTileBytes; };
      auto begin_version = [&]() {       // plain query tile -> buffer of version n_made (one thread asks the copy engine)
        if (r == 0) {
          mbar_arrive_expect_tx(&ctrl->qraw_full[t], L::kTileBytes);
          for (int c = 0; c < L::kChunks; ++c)
            tma_load_3d(ver_buf(n_made) + c * L::kRegionBytes, &tmap_q, &ctrl->qraw_full[t], c * 64, head0,
                        it.q_row0 + t * p.tok);
        }
      };
      auto finish_version = [&](bool rotated) -> bool {
        if (!mbar_wait(&ctrl->qraw_full[t], n_made & 1, abort_flag)) return false;
        if (rotated) {
          if (r < D / 2) { cs_stage[r] = cs_next; mbar_arrive(&ctrl->cs_full[t]); }
          if (!mbar_wait(&ctrl->cs_full[t], n_staged & 1, abort_flag)) return false;
          ++n_staged;
          rotate_q_row<D>(ver_buf(n_made), ver_buf(n_made), cs_stage, p.rope_layout, thread_index_anew() & 127);
        }
        fence_proxy_async();                               // the tensor core reads through the async proxy
        __syncwarp();
        if ((tid & 31) == 0) mbar_arrive(&ctrl->qr_full[t][n_made & 1]);
        ++n_made;
        return true;
      };
      // where the version after the one for block `pc` (or after the plain one: pc < 0) starts
      auto plan_next = [&](int pc) {
        next_start = tile_end;
        if (pc >= 0) {
          const int e = __ldg(p.seg.cache_tile_cu + pc + 1) - it.ctile0;   // first tile after the block
          if (e < tile_end) next_start = min(e, cached_end);
          if (next_start < cached_end) fetch_cs(pc + 1);
        }
        prep = 0;
      };
      if (kFused && n_tiles > 0) {
        const bool first_cached = tile0 < cached_end;
        if (first_cached) { f_pc = find_cache_block(p, it.ctile0 + tile0); fetch_cs(f_pc); }
        begin_version();
        ok = finish_version(first_cached);
        if (!ok) break;
        plan_next(first_cached ? f_pc : -1);
      }

      for (int j = j0; j < n_tiles; j += solo ? 2 : 1) {
        if (r == 0) BA_TR(t, j, 0);
        ok = mbar_wait(&ctrl->s_full[t], s_uses & 1, abort_flag);
        if (!ok) break;
        ++s_uses;
        tc_fence_after();
        if (r == 0) BA_TR(t, j, 1);
        // visible columns of this tile for this row: 0 .. lim
        int lim;
        const int jt = tile0 + j;
        const bool walked = p.walk && jt < it.n_cache_tiles;
        if (jt < it.n_cache_tiles) lim = walked ? ctrl->tile_valid[(tiles_before + j) & 7] - 1 : it.cache_len - jt * kBlockN - 1;
        else lim = tok_c - (it.own_row0 + (jt - it.n_cache_tiles) * kBlockN);
        uint64_t sum2[4] = {0ull, 0ull, 0ull, 0ull};       // packed (0.f, 0.f)
        // One tile of softmax for this row over kCols key columns: 128, or 64 for a half tile (only the first
        // 64 keys were multiplied; nothing of the second half is loaded, exponentiated or handed over).
        auto tile_softmax = [&](auto cols_tag) {
          constexpr int kCols = decltype(cols_tag)::value;
          uint32_t s[kCols];
#pragma unroll
          for (int c = 0; c < kCols / 32; ++c) tmem_ld_32x32b_x32(tS + c * 32, *reinterpret_cast<uint32_t(*)[32]>(&s[c * 32]));
          tmem_wait_ld();
          if (r == 0) BA_TR(t, j, 2);
          if (lim < kCols - 1) {
#pragma unroll
            for (int c = 0; c < kCols; ++c)
              if (c > lim) s[c] = 0xff800000u;               // -inf
          }
          // row maximum by a wide tree of three-input maxima (128 -> 43 -> 15 -> 5 -> 1)
          constexpr int n1 = (kCols + 2) / 3, n2 = (n1 + 2) / 3, n3 = (n2 + 2) / 3;
          float l1[n1], l2[n2], l3[n3];
          auto mx_at = [](const float *a, int n, int i) {    // max of a[3i], a[3i+1], a[3i+2] where they exist
            return (3 * i + 2 < n) ? max3(a[3 * i], a[3 * i + 1], a[3 * i + 2])
                                   : (3 * i + 1 < n) ? fmaxf(a[3 * i], a[3 * i + 1]) : a[3 * i];
          };
          const float *sf = reinterpret_cast<const float *>(s);
#pragma unroll
          for (int i = 0; i < n1; ++i) l1[i] = mx_at(sf, kCols, i);
#pragma unroll
          for (int i = 0; i < n2; ++i) l2[i] = mx_at(l1, n1, i);
#pragma unroll
          for (int i = 0; i < n3; ++i) l3[i] = mx_at(l2, n2, i);
          float mx = l3[0];
#pragma unroll
          for (int i = 1; i < n3; ++i) mx = fmaxf(mx, l3[i]);
          const float m_new = fmaxf(m_used, mx);
          if (r == 0) BA_TR(t, j, 3);
          if (j == j0) {
            m_used = m_new;
          } else {
            const bool grow = (m_new - m_used) * sl > kRescaleThreshold;
            if (__any_sync(0xffffffffu, grow)) {
              // 1 when this row's maximum did not move (also when the row has seen no key yet)
              const float alpha = (m_new == -INFINITY) ? 1.f : ex2((m_used - m_new) * sl);
              m_used = m_new;
              l *= alpha;
#pragma unroll(kRescaleUnroll)
              for (int c = 0; c < D / 32; ++c) {
                uint32_t o[32];
                tmem_ld_32x32b_x32(tO + c * 32, o);
                tmem_wait_ld();
#pragma unroll
                for (int i = 0; i < 32; ++i) o[i] = __float_as_uint(__uint_as_float(o[i]) * alpha);
                tmem_st_32x32b_x32(tO + c * 32, o);
              }
            }
          }
          const float neg_m = (m_used == -INFINITY) ? 0.f : -m_used * sl;   // no visible key so far: every p is 0
          const uint64_t sl2 = pack2(sl, sl), negm2 = pack2(neg_m, neg_m);
          // P is handed to the MMA warp in two halves so that PV can start on the first 64 keys
          // while the second 64 are still being exponentiated.  The arithmetic is packed fp32x2.  The
          // store of the first half completes while the second half is begun.
          constexpr int kLead = kCols > 64 ? 16 : 0;       // column pairs of the second half done before the first is handed over
          uint32_t pk[32], pk1[kCols > 64 ? 32 : 1];
          auto expo = [&](int e0, uint32_t &dst, int i) {
            const uint64_t x2 = fma2(pack2(__uint_as_float(s[e0]), __uint_as_float(s[e0 + 1])), sl2, negm2);
            float x0, x1;
            unpack2(x2, x0, x1);
            const float p0 = ex2(x0), p1 = ex2(x1);
            sum2[i & 3] = add2(sum2[i & 3], pack2(p0, p1));
            __nv_bfloat162 v = __floats2bfloat162_rn(p0, p1);
            dst = *reinterpret_cast<uint32_t *>(&v);
          };
#pragma unroll
          for (int i = 0; i < 32; ++i) expo(2 * i, pk[i], i);
          tmem_st_32x32b_x32(tS, pk);
#pragma unroll
          for (int i = 0; i < kLead; ++i) expo(64 + 2 * i, pk1[i], i);
          tmem_wait_st();
          tc_fence_before();
          mbar_arrive(&ctrl->p_full[t][0]);
          if (r == 0) BA_TR(t, j, 4);
          if constexpr (kCols > 64) {
#pragma unroll
            for (int i = kLead; i < 32; ++i) expo(64 + 2 * i, pk1[i], i);
            tmem_st_32x32b_x32(tS + 32, *reinterpret_cast<uint32_t(*)[32]>(&pk1[0]));
            tmem_wait_st();
            tc_fence_before();
          }
          mbar_arrive(&ctrl->p_full[t][1]);               // (half tile: nothing to hand over, that product is skipped)
          if (r == 0) BA_TR(t, j, 5);
        };
        if ((half_last && j + 1 == n_tiles) || (kWalks && walked && lim < kBlockN / 2)) tile_softmax(std::integral_constant<int, kBlockN / 2>{});
        else tile_softmax(std::integral_constant<int, kBlockN>{});
        // P of this tile is with the tensor core: time to work on the next version of the query row
        if (kFused && next_start < tile_end) {
          const bool due = tile0 + j + 1 == next_start;    // the next tile is the first to need it
          const bool next_cached = next_start < cached_end;
          if (r == 0) BA_TR(t, j, 6);
          const bool finish = prep == 1 || (prep == 0 && due);
          if (prep == 0) { begin_version(); prep = 1; }
          if (finish) { ok = finish_version(next_cached); prep = 2; }
          if (!ok) break;
          if (r == 0) BA_TR(t, j, 7);
          if (due) { if (next_cached) ++f_pc; plan_next(next_cached ? f_pc : -1); }
        }
        float sum[8];
#pragma unroll
        for (int i = 0; i < 4; ++i) unpack2(sum2[i], sum[2 * i], sum[2 * i + 1]);
        l += ((sum[0] + sum[1]) + (sum[2] + sum[3])) + ((sum[4] + sum[5]) + (sum[6] + sum[7]));
      }

      // (the item is looked up again for the write-out: its rows need not be kept in registers through the loop)
      int q_row0, q_rows, part_row0;
      asm volatile("ld.global.nc.v2.s32 {%0, %1}, [%3];\n\tld.global.nc.s32 %2, [%3 + 20];"
                   : "=&r"(q_row0), "=&r"(q_rows), "=r"(part_row0) : "l"(p.items + 8 * (size_t)e.pair));
      if (kClustered && e.fill == 2) { q_row0 += p.tok; q_rows -= p.tok; }
      if (ok && n_tiles > 0 && !(solo && t == 1)) { ok = mbar_wait(&ctrl->o_done[t], o_uses & 1, abort_flag); ++o_uses; }
      float weight = 1.f, inv1 = 0.f;      // (solo) what O_0 and O_1 count for
      if (kSolo && solo) {                 // (a cluster's CTA has one entry)
        // group 1's maximum and sum of every row, where the other deep-ring kernel stages its output
        float2 *other = reinterpret_cast<float2 *>(smem + L::kBg + L::kTileBytes) + r;
        if (t == 1) {
          if (ok) { *other = make_float2(m_used, l); mbar_arrive(&ctrl->solo_full); }
        } else if (ok) {
          ok = mbar_wait(&ctrl->solo_full, 0, abort_flag) && mbar_wait(&ctrl->o_done[1], 0, abort_flag);
          const float2 x = *other;
          const float m = fmaxf(m_used, x.x);
          if (m != -INFINITY) { weight = ex2((m_used - m) * sl); inv1 = ex2((x.x - m) * sl); }
          l = weight * l + inv1 * x.y;
          m_used = m;
        }
      }
      if (ok && !(solo && t == 1)) {
        tc_fence_after();
        const float inv_l = l > 0.f ? 1.f / l : 0.f, inv = weight * inv_l;
        inv1 *= inv_l;
        const float lse_val = l > 0.f ? (m_used * sl + log2f(l)) * 0.6931471805599453f : -INFINITY;
        const bool partial = !kClustered && e.split >= 0;
        // Rows leave through shared memory -- the warp's quarter of the entry's own query tile, which every product has
        // read by now -- so that a store instruction writes whole rows: stores straight from the row each thread owns touch
        // 32 rows at a time and took 5000-7000 cycles a tile (seven edited blocks, 312 entries: 34.9 -> 27 us a layer).
        // Its loops stay loops: the code is passed once an entry and has been displaced by the softmax loop since, so that its
        // length is what it costs (unrolled over the columns a tile took 2700-4000 cycles from the last product; rolled, a cold
        // prompt of 7200 tokens, us over eight layers: 842 -> 782; seven edited blocks 224 -> 213; 8 x 16384 tokens 3105 -> 3000;
        // 64 queries over 32000 cached tokens 592 -> 577).
        const int thread = thread_index_anew();
        const int lane = thread & 31, quarter = (thread >> 5) & 3;
        const int q_last = q_row0 + q_rows - 1, out_head0 = e.chunk * p.hpt;
        // a row is stored only if it belongs to the item and lies inside the caller's tensors; tables that
        // describe more rows than the caller gave are reported, nothing is written past the end
        const int row_tok = q_row0 + tq * p.tok + ((quarter * 32 + lane) >> p.hpt_log2), head = out_head0 + (lane & (p.hpt - 1));
        const bool row_valid = row_tok <= q_last && row_tok < p.n_q_rows;
        if (row_tok <= q_last && row_tok >= p.n_q_rows) ba_record_status(p.status, BA_ERR_SHAPE);
        // (kDeepRing: through rows of its own, 128 bytes at a time)
        constexpr int kStageRow = kDeep ? 128 : 2 * D;
        uint8_t *stage = (kDeep ? smem + L::kBg + L::kTileBytes + t * (128 * kStageRow)
                          : kFused              ? ver_buf(n_made - 1)
                                                : smem + ((p.q_double && (n_loaded & 1)) ? L::kBg + t * L::kTileBytes : (t ? L::kQ1 : L::kQ0))) +
                         quarter * (32 * kStageRow);
        // partial results of a prefill are indexed by the row's place among the rows of final blocks
        const int part_shift = partial && !p.final_only ? part_row0 - q_row0 : 0;
        const int tile_row0 = q_row0 + tq * p.tok, tile_rows = min(q_last + 1, p.n_q_rows) - tile_row0;   // tokens stored
        const size_t out_row0 = (size_t)(tile_row0 + part_shift) * p.Hq + out_head0;
        // dst: where the staged bytes of the tile's first row go; row_bytes: from one (token, head) row to the next
        auto store_rows = [&](uint8_t *dst, int row_bytes) {
          constexpr int kRowChunks = kStageRow / 16;
          const int c = lane % kRowChunks;
          dst += c * 16;
          __syncwarp();
#pragma unroll 8
          for (int i = 0; i < kRowChunks; ++i) {
            const int lr = i * (32 / kRowChunks) + lane / kRowChunks, rr = quarter * 32 + lr, tk = rr >> p.hpt_log2;
            const uint4 x = *reinterpret_cast<const uint4 *>(stage + lr * (kRowChunks * 16) + ((c ^ (lr & 7)) << 4));
            if (tk < tile_rows) *reinterpret_cast<uint4 *>(dst + (tk * p.Hq + (rr & (p.hpt - 1))) * row_bytes) = x;
          }
          __syncwarp();
        };
        // A whole tile of bf16 rows leaves as one copy, laid out in the query tile's place the way the query tile was: the
        // threads only fill shared memory (row by row as below a tile takes about 3500 cycles).
        const bool whole_tile = kVariant == kPlain && n_tiles > 0 && !partial && !p.out_f32 && tile_rows >= p.tok;
        if (whole_tile) {
          uint8_t *tile = smem + ((p.q_double && (n_loaded & 1)) ? L::kBg + t * L::kTileBytes : (t ? L::kQ1 : L::kQ0));
          uint8_t *row = tile + (thread & 127) * 128;
#pragma unroll 1
          for (int c = 0; c < D / 32; ++c) {
            uint32_t o[32];
            tmem_ld_32x32b_x32(tO + c * 32, o);
            tmem_wait_ld();
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              uint32_t w[4];
#pragma unroll
              for (int e2 = 0; e2 < 4; ++e2) {
                __nv_bfloat162 v = __floats2bfloat162_rn(__uint_as_float(o[8 * i + 2 * e2]) * inv,
                                                         __uint_as_float(o[8 * i + 2 * e2 + 1]) * inv);
                w[e2] = *reinterpret_cast<uint32_t *>(&v);
              }
              *reinterpret_cast<uint4 *>(row + (c >> 1) * L::kRegionBytes + ((((c & 1) * 4 + i) ^ (lane & 7)) << 4)) =
                  make_uint4(w[0], w[1], w[2], w[3]);
            }
          }
          fence_proxy_async();
          mbar_arrive(&ctrl->out_staged[t]);
          if ((thread & 127) == 0) {
            ok = mbar_wait(&ctrl->out_staged[t], ctrl->n_staged_out[t] & 1, abort_flag);
            ctrl->n_staged_out[t] += 1;
            if (ok) {
              for (int c = 0; c < L::kChunks; ++c) tma_store_3d(&tmap_o, tile + c * L::kRegionBytes, c * 64, out_head0, tile_row0);
              bulk_commit_group();
              out_pending = p.q_double ? (n_loaded & 1) : 0;
            }
          }
          __syncwarp();
          if (!p.q_double) release_out();                  // the next entry's queries want the same place
        } else if (kClustered) {
          // fp32 rows stay here for the other CTAs of the cluster: tile 0 over both query tiles, tile 1 over the ring (every
          // product that reads them has completed)
          if (n_tiles > 0) {
            uint8_t *row = smem + (t ? L::kRing : L::kQ0) + (thread & 127) * (D * 4);
#pragma unroll 1
            for (int c = 0; c < D / 32; ++c) {
              uint32_t a[32];
              float o[32];
              tmem_ld_32x32b_x32(tO + c * 32, a);
              tmem_wait_ld();
#pragma unroll
              for (int i = 0; i < 32; ++i) o[i] = __uint_as_float(a[i]) * inv;
              if (kSolo && solo) {
                tmem_ld_32x32b_x32(tO + 128 + c * 32, a);
                tmem_wait_ld();
#pragma unroll
                for (int i = 0; i < 32; ++i) o[i] = fmaf(__uint_as_float(a[i]), inv1, o[i]);
              }
#pragma unroll
              for (int i = 0; i < 8; ++i)
                *reinterpret_cast<float4 *>(row + (((c * 8 + i) ^ (lane & 7)) << 4)) = make_float4(o[4 * i], o[4 * i + 1], o[4 * i + 2], o[4 * i + 3]);
            }
          }
          reinterpret_cast<float *>(smem + L::kCtrl + 1024)[t * 128 + (thread & 127)] = lse_val;
        } else if (n_tiles > 0) {
          if (partial || p.out_f32) {
            uint8_t *base = partial ? reinterpret_cast<uint8_t *>(p.o_part + (size_t)e.split * p.n_part_rows * p.Hq * D)
                                    : reinterpret_cast<uint8_t *>(p.o);
#pragma unroll 1
            for (int h = 0; h < 4 * D / kStageRow; ++h) {            // kStageRow bytes of every row at a time
#pragma unroll 1
              for (int q = 0; q < kStageRow / 128; ++q) {
                uint32_t o[32];
                tmem_ld_32x32b_x32(tO + h * (kStageRow / 4) + q * 32, o);
                tmem_wait_ld();
#pragma unroll
                for (int i = 0; i < 8; ++i)
                  *reinterpret_cast<float4 *>(stage + lane * kStageRow + (((q * 8 + i) ^ (lane & 7)) << 4)) =
                      make_float4(__uint_as_float(o[4 * i]) * inv, __uint_as_float(o[4 * i + 1]) * inv,
                                  __uint_as_float(o[4 * i + 2]) * inv, __uint_as_float(o[4 * i + 3]) * inv);
              }
              store_rows(base + out_row0 * D * 4 + h * kStageRow, D * 4);
            }
          } else {
#pragma unroll 1
            for (int h = 0; h < 2 * D / kStageRow; ++h) {
#pragma unroll 1
              for (int c = 0; c < kStageRow / 64; ++c) {
                uint32_t o[32];
                tmem_ld_32x32b_x32(tO + h * (kStageRow / 2) + c * 32, o);
                tmem_wait_ld();
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                  uint32_t w[4];
#pragma unroll
                  for (int e2 = 0; e2 < 4; ++e2) {
                    __nv_bfloat162 v = __floats2bfloat162_rn(__uint_as_float(o[8 * i + 2 * e2]) * inv,
                                                             __uint_as_float(o[8 * i + 2 * e2 + 1]) * inv);
                    w[e2] = *reinterpret_cast<uint32_t *>(&v);
                  }
                  *reinterpret_cast<uint4 *>(stage + lane * kStageRow + (((c * 4 + i) ^ (lane & 7)) << 4)) = make_uint4(w[0], w[1], w[2], w[3]);
                }
              }
              store_rows(reinterpret_cast<uint8_t *>(p.o) + out_row0 * D * 2 + h * kStageRow, D * 2);
            }
          }
        }
        if (n_tiles > 0) {
          // O_t has been read out of tensor memory: the next item's first PV may overwrite it
          tc_fence_before();
          mbar_arrive(&ctrl->o_free[t]);
          if (kVariant == kPlain && !whole_tile) {
            fence_proxy_async();                           // the copy engine writes the buffer next
            __syncwarp();
            if (lane == 0) mbar_arrive(&ctrl->q_empty[p.q_double ? (n_loaded & 1) : 0][t]);
          }
        }
        if (row_valid && !kClustered) {
          float *lp = p.lse_part + (size_t)(row_tok + part_shift) * p.Hq + head;
          if (partial) {
            lp[(size_t)e.split * p.n_part_rows * p.Hq] = lse_val;
            for (int s = e.fill; s < p.n_splits; ++s)      // slots no entry of this item writes: empty
              lp[(size_t)s * p.n_part_rows * p.Hq] = -INFINITY;
          } else {
            if (p.lse) p.lse[(size_t)row_tok * p.Hq + head] = lse_val;
            if (stream && p.n_splits > 1) *lp = __uint_as_float(kRowIsComplete);
          }
        }
      }
      }
      tiles_before += n_tiles;
      if (n_tiles > 0) ++n_loaded;
      if (kClustered) break;
    }
    release_out();                        // no copy reads this CTA's memory when it ends
    if (kClustered) {
      __syncwarp();
      cluster_sync();
      const WorkEntry e = ctrl->work_ring[0];
      if (e.pair >= 0) cluster_merge_rows<D>(p, e, warp, smem_u32(smem + L::kQ0), smem_u32(smem + L::kRing), smem_u32(smem + L::kCtrl + 1024));
      __syncwarp();
    }
  }

  if (kClustered) { __syncwarp(); cluster_sync(); }       // no CTA leaves while another reads its rows
  tc_fence_before();
  __syncthreads();
  if (tid == 0) {
    if (ctrl->abort_flag) ba_record_status(p.status, BA_ERR_TIMEOUT);
    if (p.counters) {
      // every role of this CTA is done with the counters; the CTA that finishes last puts them back to zero
      __threadfence();
      if (atomicAdd(p.counters + 2, 1) == (int)gridDim.x - 1) {
        p.counters[0] = 0; p.counters[1] = 0;
        __threadfence();
        p.counters[2] = 0;
      }
    }
  }
  if (warp == 9) tmem_dealloc(tmem, 512);
}

// Merge of split-KV partial results: o = sum_s w_s o_s / sum_s w_s with w_s = exp(lse_s - max lse).
// blockIdx.y is a work item, blockIdx.x a head chunk and a part of the 256 (token, head) rows it has; one thread per 4
// columns of a row; the order of the sum is fixed, so results are run-to-run stable.  Bound by latency: the log-sum-exps of all slots are loaded before the first use, and the partial rows kBatch at
// a time (one by one, ten slots of 64 rows took 5.9 us).  In a stream launch many items need nothing and
// their CTAs leave after one load: with many items a CTA takes 32 rows (16 requests: 18 us with a CTA for every 8 rows), with
// few 8 rows at once.
struct CombineParams {
  const float *o_part, *lse_part;
  void *o;
  float *lse;
  const int32_t *items, *totals;
  int final_only, Hq, hpt, hpt_log2, parts_log2, n_part_rows, n_q_rows, n_splits, out_f32;
};
template <int D, int kMax>
__global__ void __launch_bounds__(256)
ba_combine_splits_kernel(const CombineParams p) {
  constexpr int kVec = D / 4, kBatch = kMax < 8 ? kMax : 8;
  ba_pdl_wait();
  ba_pdl_trigger();
  const int n_final = __ldg(p.totals + 3), valid = __ldg(p.totals + 7);
  const bool fit = partials_fit(p.totals, p.final_only, p.n_splits, p.n_part_rows);
  if (valid != BA_TABLES_VALID || (int)blockIdx.y >= n_final || !fit) return;    // (not valid, no room: nothing was attended either)
  const int32_t *line = p.items + 8 * ((p.final_only ? 0 : __ldg(p.totals + 2) - n_final) + blockIdx.y);
  const int q_row0 = __ldg(line), q_rows = min(__ldg(line + 1), p.n_q_rows - q_row0);
  const int part0 = p.final_only ? q_row0 : __ldg(line + 5), head0 = (blockIdx.x >> p.parts_log2) * p.hpt;
  const size_t slot = (size_t)p.n_part_rows * p.Hq;
  const int v = threadIdx.x % kVec;
  const int rows = 256 >> p.parts_log2, part_row0 = (blockIdx.x & ((1 << p.parts_log2) - 1)) * rows;
  for (int r = threadIdx.x / kVec; r < rows; r += 256 / kVec) {          // head r % hpt of token r / hpt
    const int row = (part_row0 + r) >> p.hpt_log2, h = head0 + (r & (p.hpt - 1));
    if (row >= q_rows) return;
    const size_t at = (size_t)(part0 + row) * p.Hq + h, out = (size_t)(q_row0 + row) * p.Hq + h;
    float ls[kMax], mx = -INFINITY, den = 0.f;
#pragma unroll
    for (int s = 0; s < kMax; ++s) ls[s] = s < p.n_splits ? __ldg(p.lse_part + s * slot + at) : -INFINITY;
    if (__float_as_uint(ls[0]) == kRowIsComplete) return;                // (the whole item is)
#pragma unroll
    for (int s = 0; s < kMax; ++s) mx = fmaxf(mx, ls[s]);
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int s0 = 0; s0 < kMax; s0 += kBatch) {
      float4 x[kBatch];
#pragma unroll
      for (int i = 0; i < kBatch; ++i)                       // an empty slot holds no values at all
        x[i] = ls[s0 + i] == -INFINITY ? make_float4(0.f, 0.f, 0.f, 0.f)
                                       : __ldcs(reinterpret_cast<const float4 *>(p.o_part + ((s0 + i) * slot + at) * D) + v);
#pragma unroll
      for (int i = 0; i < kBatch; ++i) {
        const float w = ls[s0 + i] == -INFINITY ? 0.f : __expf(ls[s0 + i] - mx);
        den += w;
        acc.x = fmaf(w, x[i].x, acc.x); acc.y = fmaf(w, x[i].y, acc.y); acc.z = fmaf(w, x[i].z, acc.z); acc.w = fmaf(w, x[i].w, acc.w);
      }
    }
    const float inv = 1.f / den;
    acc.x *= inv; acc.y *= inv; acc.z *= inv; acc.w *= inv;
    if (p.out_f32) {
      reinterpret_cast<float4 *>(reinterpret_cast<float *>(p.o) + out * D)[v] = acc;
    } else {
      __nv_bfloat162 a = __floats2bfloat162_rn(acc.x, acc.y), b = __floats2bfloat162_rn(acc.z, acc.w);
      uint2 w2 = make_uint2(*reinterpret_cast<uint32_t *>(&a), *reinterpret_cast<uint32_t *>(&b));
      reinterpret_cast<uint2 *>(reinterpret_cast<__nv_bfloat16 *>(p.o) + out * D)[v] = w2;
    }
    if (p.lse && v == 0) p.lse[out] = mx + logf(den);
  }
}

// ------------------------------------------------------------------ host side
typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                  const cuuint64_t *, const cuuint32_t *, const cuuint32_t *,
                                  CUtensorMapInterleave, CUtensorMapSwizzle, CUtensorMapL2promotion,
                                  CUtensorMapFloatOOBfill);

EncodeTiledFn encode_fn() {
  static EncodeTiledFn fn = nullptr;
  if (!fn) {
    void *p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) != cudaSuccess) return nullptr;
    fn = reinterpret_cast<EncodeTiledFn>(p);
  }
  return fn;
}

// [rows, heads, d] bf16 viewed as a 3-D tensor (d, head, row); box = 64 columns x box_heads x box_rows, 128-byte swizzle.
bool make_map(CUtensorMap *m, const void *ptr, int D, int heads, long long rows, int box_heads, int box_rows) {
  EncodeTiledFn enc = encode_fn();
  if (!enc || rows < 1) return false;
  cuuint64_t dims[3] = {(cuuint64_t)D, (cuuint64_t)heads, (cuuint64_t)rows};
  cuuint64_t strides[2] = {(cuuint64_t)D * 2, (cuuint64_t)heads * D * 2};
  cuuint32_t box[3] = {64, (cuuint32_t)box_heads, (cuuint32_t)box_rows};
  cuuint32_t es[3] = {1, 1, 1};
  // A row of a head is read in 128-byte boxes; with D = 128 the first brings the whole 256 bytes into L2 (timed in turn with 128
  // bytes: 32 layers of 768 queries over 32000 cached tokens 13000 -> 12920 us, 64 queries 607 -> 605; pooled requests
  // 1311 -> 1323, prefills the same; two runs of one side differ by up to 0.6 %).
  return enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void *>(ptr), dims, strides, box, es,
             CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, D == 128 ? CU_TENSOR_MAP_L2_PROMOTION_L2_256B : CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
             CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

}  // namespace

// Tensor maps of the tensors recently passed to the attention calls.  A serving loop hands the same
// few buffers to the library layer after layer; encoding a map costs a driver call each time, so
// the maps are kept in a small direct-mapped table keyed by everything that goes into them.
struct ba_map_cache {
  static constexpr int kSlots = 512;
  struct Slot {
    const void *ptr;
    long long rows;
    int D, heads, box_heads, box_rows;
    alignas(64) CUtensorMap map;
  } slot[kSlots];
};

namespace {

// (by value: two tensors of one call can share a slot)
bool cached_map(ba_ctx *ctx, CUtensorMap *out, const void *ptr, int D, int heads, long long rows, int box_heads, int box_rows) {
  uint64_t h = (uint64_t)(uintptr_t)ptr * 0x9E3779B97F4A7C15ull;
  h ^= (uint64_t)rows * 0xC2B2AE3D27D4EB4Full + (uint64_t)(box_heads * 131 + box_rows);
  ba_map_cache::Slot &sl = ctx->maps->slot[(h >> 40) & (ba_map_cache::kSlots - 1)];
  if (sl.ptr != ptr || sl.rows != rows || sl.D != D || sl.heads != heads || sl.box_heads != box_heads || sl.box_rows != box_rows) {
    sl.ptr = nullptr;
    if (!make_map(&sl.map, ptr, D, heads, rows, box_heads, box_rows)) return false;
    sl.ptr = ptr; sl.rows = rows; sl.D = D; sl.heads = heads; sl.box_heads = box_heads; sl.box_rows = box_rows;
  }
  *out = sl.map;
  return true;
}

template <int D>
constexpr int attend_smem_bytes() {
  // ask for more than half of the SM's shared memory so that two CTAs never share an SM
  // (each CTA allocates all 512 tensor-memory columns)
  return Layout<D>::kBytes + 1024 > 120 * 1024 ? Layout<D>::kBytes + 1024 : 120 * 1024;
}

}  // namespace

// Per-context set-up of the attention path, with the context's device current: the kernels' shared-memory
// limit is raised once here instead of on every launch, and the tensor-map table is created.
ba_status ba_attend_sm100_setup(ba_ctx *ctx) {
  auto raise = [](auto kern, int bytes) { return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes); };
  // (The kernels lie in memory in the reverse of this order, and one that moves gains or loses up to 1 % with the same code: five
  // orders, us a pass, cold prompt of 7200 tokens 767-772, 32 x 1000 cached tokens and one final token 479-490; 765 and 489 without
  // kSharedCluster, 767 and 483 with it last in memory, where it moves no other kernel.)
  BA_CUDA_TRY(raise(ba_attend_sm100_kernel<128, kSharedCluster>, attend_smem_bytes<128>()));
  BA_CUDA_TRY(raise(ba_attend_sm100_kernel<64, kSharedCluster>, attend_smem_bytes<64>()));
  BA_CUDA_TRY(raise(ba_attend_sm100_kernel<128, kPlain>, attend_smem_bytes<128>()));
  BA_CUDA_TRY(raise(ba_attend_sm100_kernel<128, kFusedPath>, attend_smem_bytes<128>()));
  BA_CUDA_TRY(raise(ba_attend_sm100_kernel<128, kDeepRing>, attend_smem_bytes<128>()));
  BA_CUDA_TRY(raise(ba_attend_sm100_kernel<128, kFusedCluster>, attend_smem_bytes<128>()));
  BA_CUDA_TRY(raise(ba_attend_sm100_kernel<128, kDeepCluster>, attend_smem_bytes<128>()));
  BA_CUDA_TRY(raise(ba_attend_sm100_kernel<64, kPlain>, attend_smem_bytes<64>()));
  BA_CUDA_TRY(raise(ba_attend_sm100_kernel<64, kFusedPath>, attend_smem_bytes<64>()));
  BA_CUDA_TRY(raise(ba_attend_sm100_kernel<64, kDeepRing>, attend_smem_bytes<64>()));
  BA_CUDA_TRY(raise(ba_attend_sm100_kernel<64, kFusedCluster>, attend_smem_bytes<64>()));
  BA_CUDA_TRY(raise(ba_attend_sm100_kernel<64, kDeepCluster>, attend_smem_bytes<64>()));
  ctx->maps = new (std::nothrow) ba_map_cache();
  if (!ctx->maps) return BA_ERR_CUDA;
  for (auto &sl : ctx->maps->slot) sl.ptr = nullptr;
  return BA_OK;
}

void ba_attend_sm100_teardown(ba_ctx *ctx) {
  delete ctx->maps;
  ctx->maps = nullptr;
}

// Diagnostic: one CTA waits on an mbarrier that nothing ever arrives on, with the same bounded
// wait the attention kernel uses, so the expiry path (abort flag, status word, clean return) can be
// checked on a live device without any fault.
__global__ void ba_wait_expiry_kernel(int32_t *status) {
  __shared__ uint64_t bar;
  __shared__ int abort_flag;
  if (threadIdx.x == 0) { mbar_init(&bar, 1); abort_flag = 0; fence_barrier_init(); }
  __syncthreads();
  const bool ok = mbar_wait(&bar, 0, &abort_flag);       // never completes: gives up after the poll limit
  __syncthreads();
  if (threadIdx.x == 0 && (!ok || abort_flag)) ba_record_status(status, BA_ERR_TIMEOUT);
}

extern "C" ba_status ba_selftest_wait_expiry(ba_ctx *ctx, void *stream) {
  if (!ctx) return BA_ERR_INVALID_ARG;
  BA_CUDA_TRY(cudaSetDevice(ctx->device));
  ba_wait_expiry_kernel<<<1, 64, 0, (cudaStream_t)stream>>>(ctx->dev_status);
  BA_CUDA_TRY(cudaGetLastError());
  ctx->launches += 1;
  return BA_OK;
}

// Clusters of n attention CTAs (one per SM) the device runs at a time; asked once per process, device and size.
static int max_clusters(ba_ctx *ctx, int n) {
  static std::atomic<int> known[64][kMaxCluster + 1];
  std::atomic<int> &slot = known[ctx->device & 63][n];
  int v = slot.load(std::memory_order_relaxed);
  if (v == 0) {
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = (unsigned)n; attr.val.clusterDim.y = 1; attr.val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(ctx->sm_count / n * n)); cfg.blockDim = dim3(kThreads); cfg.dynamicSmemBytes = attend_smem_bytes<128>();
    cfg.attrs = &attr; cfg.numAttrs = 1;
    int got = 0;
    if (cudaOccupancyMaxActiveClusters(&got, ba_attend_sm100_kernel<128, kDeepCluster>, &cfg) != cudaSuccess) { cudaGetLastError(); got = 0; }
    v = got + 1;
    slot.store(v, std::memory_order_relaxed);
  }
  return v - 1;
}

// Heads of one KV group packed into a query tile: the largest of 4, 2, 1 that divides the group size.
int ba_heads_per_tile(const ba_config &c) {
  int G = c.n_q_heads / c.n_kv_heads;
  return (G % 4 == 0) ? 4 : (G % 2 == 0) ? 2 : 1;
}

// The fused call in two steps: re-encode the cached keys into k_out, or the end of the workspace, and attend them.  The fused
// kernel rotates every query tile once per cached block and cannot let a key tile span two blocks.  Taken
//  * when k_out is wanted: the keys are read twice otherwise (32 x 1000 cached tokens and a final block of 1 / 64 / 128: 76 / 88 /
//    119 us with the re-encoding beside the fused kernel, 67 / 73 / 100 in two steps; paged 79 / 92 / 125 and 72 / 80 / 109);
//  * with more than one pair of query tiles per sequence (8 requests, 29000 cached tokens in blocks of 37-611, final blocks of
//    64 / 101 / 256 tokens: fused 81 / 121 / 244 us, two steps 74 / 95 / 163);
//  * for caches a re-encoding pass takes only a few microseconds over (10 x 128-384 and 32: 23.5 and 19.9).
// What is left to the fused kernel: short final blocks over long caches (32 x 1000 and 1 / 32 / 64: 53 / 55 / 66 us, two steps
// 67 / 68 / 73), and rows wider than the re-encoding kernel takes.
static bool fused_in_two_steps(const ba_ctx *ctx, const ba_attend_args &a, const ba_segments *seg, size_t *scratch) {
  if (!a.fused || !a.final_only || a.n_cache_rows < 1 || !seg->cache_rope) return false;
  if (a.k_out) return true;
  if (ba_reencode_units(ctx->cfg.rope_layout, ctx->cfg.n_kv_heads * ctx->cfg.head_dim / 8) > kBaReencodeMaxUnits) return false;
  *scratch = ba_align_up((size_t)a.n_cache_rows * ctx->cfg.n_kv_heads * ctx->cfg.head_dim * 2, 256);
  if (*scratch > (16u << 20) && (seg->n_final_items < 1 || 2LL * seg->n_final_items < 3LL * seg->batch)) return false;
  return ctx->workspace && ctx->workspace_bytes > ba_scratch_offset(ctx) && *scratch <= (ctx->workspace_bytes - ba_scratch_offset(ctx)) / 2;
}

ba_status ba_attend_sm100_launch(ba_ctx *ctx, const ba_attend_args &a, const ba_segments *seg,
                                 cudaStream_t stream) {
  size_t scratch = 0;
  if (fused_in_two_steps(ctx, a, seg, &scratch)) {
    ba_status st = ba_flush_pending(ctx, stream);
    if (st != BA_OK) return st;
    ba_attend_args b = a;
    b.fused = 0; b.k_src_off = nullptr; b.k_out = nullptr;
    b.reserved_bytes = a.k_out ? 0 : scratch;
    void *keys = a.k_out ? a.k_out : (char *)ctx->workspace + (ctx->workspace_bytes - scratch) / 256 * 256;
    b.k_cache = (const __nv_bfloat16 *)keys;
    ba_reencode_job job = ba_make_reencode_job(ctx, a.k_cache, a.k_src_off, a.n_k_rows, keys, seg->cache_cu, seg->cache_delta,
                                               seg->n_cached_blocks, a.n_cache_rows, reinterpret_cast<const float2 *>(seg->cache_rope));
    // A row outside the source is a row of zeros for the attention, as the fused kernel's loads have it; nothing that k_out or
    // the workspace held before may show.  Only written keys are reported: those are ba_reencode_k's.
    job.totals = seg->totals;
    job.outside = a.k_out ? BA_ROWS_ZERO_REPORTED : BA_ROWS_ZERO;
    if (a.page_rows > 0) {
      job.src_off = nullptr; job.page_cu = a.page_cu; job.page_idx = a.page_idx;
      while ((1 << job.page_lg) < a.page_rows) ++job.page_lg;
    }
    st = ba_reencode_main_launch(ctx, job, stream);
    return st == BA_OK ? ba_attend_sm100_launch(ctx, b, seg, stream) : st;
  }
  const int D = ctx->cfg.head_dim, Hq = ctx->cfg.n_q_heads, Hkv = ctx->cfg.n_kv_heads;
  AttnParams p;
  p.o = a.o; p.lse = a.lse; p.status = ctx->dev_status; p.out_f32 = a.out_f32;
  p.Hq = Hq; p.Hkv = Hkv; p.G = Hq / Hkv;
  p.hpt = ba_heads_per_tile(ctx->cfg);
  p.hpt_log2 = p.hpt == 4 ? 2 : p.hpt == 2 ? 1 : 0;
  p.tok = 128 / p.hpt;
  p.scale = ctx->scale;
  p.scale_log2 = ctx->scale * 1.4426950408889634f;
  p.final_only = a.final_only;
  p.balanced = 0; p.bal_len = 0; p.q_double = 0;
  p.v_src_off = a.final_only ? a.v_src_off : nullptr;
  p.fused = a.final_only && a.fused && a.n_cache_rows > 0;
  p.k_src_off = p.fused ? a.k_src_off : nullptr;
  p.page_cu = nullptr; p.page_idx = nullptr; p.page_lg = 0; p.k_paged = 0; p.v_paged = 0;
  if (a.final_only && a.page_rows > 0 && a.n_cache_rows > 0) {
    p.page_cu = a.page_cu; p.page_idx = a.page_idx;
    while ((1 << p.page_lg) < a.page_rows) ++p.page_lg;
    p.v_paged = 1;
    p.k_paged = p.fused ? 1 : 0;
    p.v_src_off = nullptr; p.k_src_off = nullptr;
  }
  p.walk = p.v_src_off != nullptr || p.fused || p.v_paged;
  p.rope_layout = ctx->cfg.rope_layout;
  p.q_rope = p.fused ? reinterpret_cast<const float2 *>(seg->cache_rope) : nullptr;
  if (p.fused && !p.q_rope) return BA_ERR_INVALID_ARG;
  p.n_q_rows = a.n_q_rows;
  p.seg = *seg;
  p.items = a.final_only ? seg->final_items : seg->prompt_items;
  if (!p.items) return BA_ERR_INVALID_ARG;
  if (seg->q_tile_tokens != 2 * p.tok) return BA_ERR_INVALID_ARG;

  // Split the keys of each work item over several CTAs when the items alone cannot fill the
  // GPU (a short final block over a long cache).  The split count minimises
  // waves x (tiles per CTA + a fixed per-CTA cost) and is capped by the workspace.
  const int pair_tok = 2 * p.tok;
  const int n_units = a.final_only ? seg->batch : seg->n_blocks;
  // work items: the exact count when ba_segment() saw the lengths on the host, else an upper bound
  const int pairs_known = a.final_only ? seg->n_final_items : seg->n_prompt_items;
  const unsigned pairs_upper = pairs_known > 0 ? (unsigned)pairs_known : (unsigned)(a.n_q_rows / pair_tok + n_units);
  const long long items = (a.final_only && seg->n_final_items > 0 ? (long long)seg->n_final_items
                                                                  : (long long)((a.n_q_rows + pair_tok - 1) / pair_tok)) * (Hq / p.hpt);
  int n_splits = 1, stream_ctas = 0, cluster_shared = 0;
  p.stream = 0; p.n_odd = 0; p.cluster = 0; p.single = 0;
  if (a.final_only) {
    // key tiles of an average item: counted by ba_segment() when it saw the lengths, else estimated
    const int32_t *ft = seg->final_key_tiles + (p.walk ? 3 : 0);
    const long long avg_tiles = (ft[0] > 0 && seg->n_final_items > 0)
                                    ? (ft[0] + seg->n_final_items - 1) / seg->n_final_items
                                    : ((long long)a.n_cache_rows / seg->batch + pair_tok) / kBlockN + 1;
    const size_t per_split = (size_t)a.n_q_rows * Hq * (D + 1) * sizeof(float);
    // the angle table of a queued re-encoding job sits at the end of the workspace and is read by
    // this very launch: the partial results must stay below it
    const size_t taken = ba_scratch_offset(ctx) + ctx->pending_table_bytes + (a.reserved_bytes ? a.reserved_bytes + 256 : 0);
    const size_t avail = ctx->workspace_bytes > taken ? ctx->workspace_bytes - taken : 0;
    const int cap = (int)min((size_t)32, per_split ? avail / per_split : 0);
    // equal splits or the balanced launch (ba_plan_splits, above the kernels' common declarations)
    const ba_split_plan plan = ba_plan_splits(ctx->sm_count, items, seg->n_final_items, Hq / p.hpt, avg_tiles, ft, cap);
    n_splits = plan.n_splits; p.balanced = plan.balanced; p.bal_len = plan.bal_len;
    if (!p.balanced && ft[0] > 0 && cap > 0) {
      const ba_stream_plan stream = ba_plan_stream(ctx->sm_count, Hq / p.hpt, ft, seg->final_key_tiles_odd[p.walk ? 1 : 0], cap);
      const long long equal_cost = ba_equal_splits_cost(ctx->sm_count, items, ft[2], n_splits);
      if (stream.n_ctas > 0 && stream.cost < equal_cost) {
        p.stream = 1; stream_ctas = stream.n_ctas; p.n_odd = stream.n_odd; n_splits = stream.n_slots;
      }
      if (a.n_cache_rows > 0 && !ctx->has_pending) {
        const ba_cluster_plan cl = ba_plan_cluster(items, a.n_q_rows > (long long)p.tok * seg->n_final_items,
                                                   seg->final_rows_max > 0 && seg->final_rows_max <= p.tok, p.fused, ft[2], [&](int n) { return max_clusters(ctx, n); });
        if (cl.size > 0 && cl.cost < (double)(p.stream ? stream.cost : equal_cost)) { p.cluster = cl.size; p.single = cl.single; cluster_shared = cl.shared; p.stream = 0; n_splits = 1; }
      }
    }
  } else if (!a.final_only && a.mode == BA_MODE_BLOCK && seg->n_final_items > 0 && seg->prompt_key_tiles > 0) {
    // The items of final blocks see the whole prompt: with few of them the launch would end on one CTA each.
    const size_t per_split = (size_t)seg->n_final_items * pair_tok * Hq * (D + 1) * sizeof(float);
    const size_t taken = ba_scratch_offset(ctx) + ctx->pending_table_bytes;
    const size_t avail = ctx->workspace_bytes > taken ? ctx->workspace_bytes - taken : 0;
    n_splits = ba_plan_final_splits(ctx->sm_count, Hq / p.hpt, seg->n_prompt_items, seg->prompt_key_tiles,
                                    seg->final_key_tiles[2], (int)min((size_t)16, avail / per_split));
  }
  p.n_splits = n_splits;
  p.n_chunks = Hq / p.hpt;
  // More entries than SMs: persistent CTAs, one per SM, draw entries from a counter, which hides each
  // entry's start-up and write-out behind its neighbours (cold prefill: many entries per SM; final block
  // over a long cache: about two, the write-out of a CTA's first entry overlaps the start of its second).
  // Shorter lists are launched one CTA per entry.
  const long long work_upper = ((long long)pairs_upper * (a.final_only ? n_splits : 1) +
                                (a.final_only ? 0 : (long long)seg->n_final_items * (n_splits - 1))) * (Hq / p.hpt);
  p.persistent = !p.balanced && !p.stream && p.cluster <= 1 && work_upper > ctx->sm_count;
  // the counters live in the last 256 bytes below the scratch area: zeroed by ba_create, left at zero by every launch
  int32_t *counters = nullptr;
  if (ctx->workspace && ctx->workspace_bytes >= ba_scratch_offset(ctx))
    counters = ba_counters(ctx);
  p.counters = nullptr;
  if (p.persistent && !counters) p.persistent = 0;   // a context without workspace: one CTA per entry, however many
  if (p.persistent) p.counters = counters;
  p.o_part = nullptr; p.lse_part = nullptr;
  p.n_part_rows = a.final_only ? a.n_q_rows : seg->n_final_items * pair_tok;
  if (n_splits > 1) {
    p.o_part = reinterpret_cast<float *>(reinterpret_cast<char *>(ctx->workspace) + ba_scratch_offset(ctx));
    p.lse_part = p.o_part + (size_t)n_splits * p.n_part_rows * Hq * D;
  }

  CUtensorMap tq, tk, tv;
  if (!cached_map(ctx, &tq, a.q, D, Hq, a.n_q_rows, p.hpt, p.tok) || !cached_map(ctx, &tk, a.k, D, Hkv, a.n_kv_rows, 1, kBlockN) ||
      !cached_map(ctx, &tv, a.v, D, Hkv, a.n_kv_rows, 1, kBlockN))
    return BA_ERR_CUDA;
  CUtensorMap tkc = tk, tvc = tv, to = tq;
  if (!a.out_f32 && !cached_map(ctx, &to, a.o, D, Hq, a.n_q_rows, p.hpt, p.tok)) return BA_ERR_CUDA;
  if (a.final_only && a.n_cache_rows > 0) {
    const int page_box = p.v_paged ? min(kBlockN, a.page_rows) : kBlockN;
    if (!cached_map(ctx, &tkc, a.k_cache, D, Hkv, p.fused ? a.n_k_rows : a.n_cache_rows, 1, p.k_paged ? page_box : kBlockN) ||
        !cached_map(ctx, &tvc, a.v_cache, D, Hkv, (a.v_src_off || p.v_paged) ? a.n_v_rows : a.n_cache_rows, 1, page_box))
      return BA_ERR_CUDA;
  }
  dim3 grid((unsigned)(p.cluster > 1 ? (items << p.single) * p.cluster : p.stream ? stream_ctas : (p.persistent || p.balanced) ? ctx->sm_count : work_upper));
  // a queued re-encoding job rides along in the spare warps; a job whose rows do not fit the
  // staging buffers is run on its own first
  p.bg.n_rows = 0; p.bg_rows_per_chunk = 0;
  if (ctx->has_pending) {
    const int row_bytes = ctx->pending.row_vecs * 16;
    if (row_bytes <= kBgStageBytes && !p.fused && counters) {   // (the fused path has other uses for the spare warps' staging area)
      p.bg = ctx->pending;
      ctx->has_pending = 0;
      ctx->pending_table_bytes = 0;
      p.bg_rows_per_chunk = kBgStageBytes / row_bytes < 32 ? kBgStageBytes / row_bytes : 32;
      p.counters = counters;
    } else {
      ba_status fs = ba_flush_pending(ctx, stream);
      if (fs != BA_OK) return fs;
    }
  }
  // The staging area is free on the plain path without a background job: a deeper ring where the keys and
  // values are streamed once or twice (final blocks over their caches; in the balanced launch a tile is read by many CTAs
  // and comes from L2), a second pair of query buffers elsewhere.
  const bool free_area = !p.fused && p.bg.n_rows == 0;
  const bool deep_ring = free_area && a.final_only && a.n_cache_rows > 0 && !p.balanced;
  p.q_double = free_area && !deep_ring;
  // (The balanced launch fills the GPU for hundreds of microseconds, and a re-encode on another stream fills the SMs it leaves
  // at its end: early CTAs of the next kernel would only take those.)
  const bool early = !p.balanced;
  cudaError_t launched = cudaSuccess;
  auto launch_attend = [&](auto kern, int smem) { launched = ba_launch_clusters(kern, p.cluster, grid, kThreads, smem, stream, early, tq, tk, tv, tkc, tvc, to, p); };
  const int variant = p.fused ? (p.cluster > 1 ? kFusedCluster : kFusedPath) : deep_ring ? (p.cluster > 1 ? (cluster_shared ? kSharedCluster : kDeepCluster) : kDeepRing) : kPlain;
  auto pick = [&](auto d_tag) {
    constexpr int kD = decltype(d_tag)::value, kSmem = attend_smem_bytes<kD>();
    switch (variant) {
      case kFusedPath: launch_attend(ba_attend_sm100_kernel<kD, kFusedPath>, kSmem); break;
      case kFusedCluster: launch_attend(ba_attend_sm100_kernel<kD, kFusedCluster>, kSmem); break;
      case kDeepRing: launch_attend(ba_attend_sm100_kernel<kD, kDeepRing>, kSmem); break;
      case kDeepCluster: launch_attend(ba_attend_sm100_kernel<kD, kDeepCluster>, kSmem); break;
      case kSharedCluster: launch_attend(ba_attend_sm100_kernel<kD, kSharedCluster>, kSmem); break;
      default: launch_attend(ba_attend_sm100_kernel<kD, kPlain>, kSmem);
    }
  };
  if (D == 128) pick(std::integral_constant<int, 128>{});
  else pick(std::integral_constant<int, 64>{});
  BA_CUDA_TRY(launched);
  ctx->launches += 1;
  ctx->last_attend[0] = (int32_t)grid.x; ctx->last_attend[1] = n_splits;
  ctx->last_attend[2] = p.balanced; ctx->last_attend[3] = p.bal_len;
  if (n_splits > 1) {
    const unsigned n_merge_items = a.final_only && seg->n_final_items == 0 ? pairs_upper : (unsigned)seg->n_final_items;
    const int parts_log2 = n_merge_items * p.n_chunks <= 64 ? 5 : 3;
    CombineParams c = {p.o_part, p.lse_part, a.o, a.lse, p.items, seg->totals, a.final_only, Hq, p.hpt, p.hpt_log2, parts_log2, p.n_part_rows,
                       a.n_q_rows, n_splits, a.out_f32};
    const dim3 cgrid((unsigned)(p.n_chunks << parts_log2), n_merge_items);
    auto launch = [&](auto kern) { launched = ba_launch(kern, cgrid, 256, 0, stream, early, c); };
    if (D == 128) {
      if (n_splits <= 4) launch(ba_combine_splits_kernel<128, 4>);
      else if (n_splits <= 8) launch(ba_combine_splits_kernel<128, 8>);
      else launch(ba_combine_splits_kernel<128, 32>);
    } else {
      if (n_splits <= 4) launch(ba_combine_splits_kernel<64, 4>);
      else if (n_splits <= 8) launch(ba_combine_splits_kernel<64, 8>);
      else launch(ba_combine_splits_kernel<64, 32>);
    }
    BA_CUDA_TRY(launched);
    ctx->launches += 1;
  }
  return BA_OK;
}
