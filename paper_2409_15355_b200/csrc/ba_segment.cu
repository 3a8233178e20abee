// Segment tables of a ragged batch (Section 2.2: one passage per block, the user
// query is the final block; Section 2.5: a block's positions follow from its
// place in the prompt; Section 2.3: cached blocks start at position zero, so the
// re-encoding delta of a block is the prompt position of its first token).
//
// The tables are a few kilobytes of integers: what this costs is latency -- launches, dependent loads, barriers -- and
// it is paid once per prompt before any layer can start.  For up to kSharedBlocks blocks everything is one launch: every
// CTA scans the block lengths on its own (all prefix sums of a scan share two barriers), keeps the block tables in shared
// memory and fills its share of the per-token, per-item and rotation tables from there; CTA 0 also writes the block
// tables.  Host-side lengths travel as kernel arguments, without a staging copy.  Larger batches run the scan as one CTA
// and the rest as a second launch.  A prompt of five blocks: two staging copies and three kernels, 12 us of GPU time and as
// many gaps, before; one kernel of 6.7 us now (a whole small request, tables included, 59 -> 40 us).
#include "ba_common.cuh"

namespace {

constexpr int kSharedBlocks = 1024;      // blocks one launch takes: one per thread, 256 or 1024 threads

// CTA-wide exclusive scans of N ints per thread at once: v[] becomes the exclusive prefixes, total[] the sums.
// `smem` holds N * 33 ints.
template <int N>
__device__ __forceinline__ void cta_exclusive_scan(int (&v)[N], int (&total)[N], int *smem) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int inc[N];
#pragma unroll
  for (int k = 0; k < N; ++k) inc[k] = v[k];
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
#pragma unroll
    for (int k = 0; k < N; ++k) {
      const int n = __shfl_up_sync(0xffffffffu, inc[k], d);
      if (lane >= d) inc[k] += n;
    }
  }
  __syncthreads();  // smem reuse across consecutive scans
  if (lane == 31) {
#pragma unroll
    for (int k = 0; k < N; ++k) smem[k * 33 + warp] = inc[k];
  }
  __syncthreads();
  if (warp < N) {
    int *row = smem + warp * 33;
    const int w = lane < (int)blockDim.x >> 5 ? row[lane] : 0;
    int winc = w;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const int n = __shfl_up_sync(0xffffffffu, winc, d);
      if (lane >= d) winc += n;
    }
    row[lane] = winc - w;  // exclusive prefix of the warp totals
    if (lane == 31) row[32] = winc;
  }
  __syncthreads();
#pragma unroll
  for (int k = 0; k < N; ++k) {
    total[k] = smem[k * 33 + 32];
    v[k] = smem[k * 33 + warp] + inc[k] - v[k];
  }
}

// First index in a[0..n) whose value is > x (a ascending).
__device__ __forceinline__ int upper_bound(const int32_t *a, int n, int x) {
  int lo = 0, hi = n;
  while (lo < hi) {
    int mid = (lo + hi) >> 1;
    if (a[mid] <= x) lo = mid + 1; else hi = mid;
  }
  return lo;
}

// The block tables the second part reads: shared memory (one launch) or the caller's table buffer (two launches).
struct BlockTables {
  int32_t *cu_seq_block, *cu_block, *cu_qtile, *kv_begin, *delta, *cache_tile_cu, *cache_delta;
  int32_t *cu_seq, *cu_final_seq, *cu_ftile;
};

struct SegmentArgs {
  int batch, B, T, mode, tile_tok, gen, half_dim;
  double neg2_over_d_log2_base;
  ba_segments seg;
  int32_t *status;
};

// Sum over the query tiles of a final block of `fin` rows of the key tiles each sees in the block itself.
__device__ __forceinline__ int own_tiles_sum(int fin, int tt) {
  const int n = (fin + tt - 1) / tt - 1;                         // whole query tiles in front of the last one
  const int whole = tt == 64 ? ((n + 1) * (n + 1)) / 4           // sum of ceil(k / 2), k = 1 .. n
                             : (n * (n + 1) / 2) * (tt >> 7);    // sum of k * tt / 128
  return whole + (fin + 127) / 128;
}

// The same over every second item (1, 3, ..): whole ones end at 2 * tt, 4 * tt, .. rows, multiples of 128.
__device__ __forceinline__ int own_tiles_sum_odd(int fin, int tt) {
  const int n = (fin + tt - 1) / tt, cut = n % 2 == 0 && fin % tt != 0, whole = n / 2 - cut;
  return (whole * (whole + 1) / 2) * (tt >> 6) + (cut ? (fin + 127) / 128 : 0);
}

// Prefix sums over blocks and sequences.  Returns false when the lengths are inconsistent.  `writer`: this CTA also
// writes the caller's tables.
template <bool kShared>
__device__ __forceinline__ bool segment_blocks(const SegmentArgs &a, const int32_t *__restrict__ lens,
                                               const int32_t *__restrict__ seq_nblocks, const BlockTables &t, bool writer,
                                               int *scan_smem, int *bad) {
  const ba_segments &seg = a.seg;
  const int tid = threadIdx.x, batch = a.batch, B = a.B, tt = a.tile_tok;
  if (tid == 0) {
    *bad = 0;
    if (writer) { seg.totals[7] = 0; seg.totals[6] = a.gen; }    // [6]: stamp of this call
  }
  __syncthreads();

  // --- first block of every sequence
  int carry = 0;
  bool seq_bad = false;
  for (int base = 0; base < batch; base += (int)blockDim.x) {
    const int s = base + tid;
    int v[1] = {s < batch ? seq_nblocks[s] : 0}, total[1];
    if (s < batch && v[0] < 1) { seq_bad = true; v[0] = 0; }
    cta_exclusive_scan<1>(v, total, scan_smem);
    if (s < batch) {
      t.cu_seq_block[s] = carry + v[0];
      if (kShared && writer) seg.cu_seq_block[s] = carry + v[0];
    }
    carry += total[0];
  }
  if (tid == 0) {
    t.cu_seq_block[batch] = carry;
    if (kShared && writer) seg.cu_seq_block[batch] = carry;
  }
  // (one decision for all threads, made before any of them can raise the flag for a block's length)
  if (__syncthreads_or(carry != B || seq_bad)) return false;

  // --- per-block prefix sums: rows, rows of final blocks, query tiles, 128-key tiles (all / final blocks), query tiles of
  // the final blocks
  int c[6] = {0, 0, 0, 0, 0, 0};
  for (int base = 0; base < B; base += (int)blockDim.x) {
    const int b = base + tid;
    int len = 0, fin = 0, s = 0, first = 0;
    if (b < B) {
      len = lens[b];
      if (len < 1) { *bad = 1; len = 0; }
      s = upper_bound(t.cu_seq_block, batch + 1, b) - 1;
      fin = b == t.cu_seq_block[s + 1] - 1;
      first = b == t.cu_seq_block[s];
    }
    const int qt = (len + tt - 1) / tt, kt = (len + 127) / 128;
    int e[6] = {len, fin ? len : 0, qt, kt, fin ? kt : 0, fin ? qt : 0}, total[6];
    cta_exclusive_scan<6>(e, total, scan_smem);
#pragma unroll
    for (int k = 0; k < 6; ++k) e[k] += c[k];
    if (b < B) {
      t.cu_block[b] = e[0];
      t.cu_qtile[b] = e[2];
      if (!fin) t.cache_tile_cu[b - s] = e[3] - e[4];            // every earlier sequence contributed exactly one final block
      if (first) t.cu_seq[s] = e[0];
      if (fin) { t.cu_final_seq[s] = e[1]; t.cu_ftile[s] = e[5]; }
      if (writer) {
        if (kShared) {
          seg.cu_block[b] = e[0]; seg.cu_qtile[b] = e[2];
          if (!fin) seg.cache_tile_cu[b - s] = e[3] - e[4];
          if (first) seg.cu_seq[s] = e[0];
          if (fin) { seg.cu_final_seq[s] = e[1]; seg.cu_ftile[s] = e[5]; }
        }
        seg.block_seq[b] = s;
        seg.block_is_final[b] = (uint8_t)fin;
        seg.block_part_off[b] = fin ? e[1] : e[0] - e[1];
        seg.cu_ktile[b] = e[3];
        if (first) seg.cu_cache_seq[s] = e[0] - e[1];
        if (!fin) { seg.cache_block[b - s] = b; seg.cache_cu[b - s] = e[0] - e[1]; }
      }
    }
#pragma unroll
    for (int k = 0; k < 6; ++k) c[k] += total[k];
  }
  if (tid == 0) {
    if (c[0] != a.T) *bad = 1;
    t.cu_block[B] = c[0]; t.cu_qtile[B] = c[2]; t.cache_tile_cu[B - batch] = c[3] - c[4];
    t.cu_seq[batch] = c[0]; t.cu_final_seq[batch] = c[1]; t.cu_ftile[batch] = c[5];
    if (writer) {
      if (kShared) {
        seg.cu_block[B] = c[0]; seg.cu_qtile[B] = c[2]; seg.cache_tile_cu[B - batch] = c[3] - c[4];
        seg.cu_seq[batch] = c[0]; seg.cu_final_seq[batch] = c[1]; seg.cu_ftile[batch] = c[5];
      }
      seg.cache_cu[B - batch] = c[0] - c[1];
      seg.cu_cache_seq[batch] = c[0] - c[1];
      seg.cu_ktile[B] = c[3];
      seg.totals[0] = c[0] - c[1]; seg.totals[1] = c[1]; seg.totals[2] = c[2]; seg.totals[3] = c[5];
    }
  }
  __syncthreads();
  if (*bad) return false;

  // --- deltas and visibility ranges
  for (int b = tid; b < B; b += (int)blockDim.x) {
    const int s = upper_bound(t.cu_seq_block, batch + 1, b) - 1;
    const int seq_start = t.cu_seq[s], start = t.cu_block[b];
    const int fin = b == t.cu_seq_block[s + 1] - 1;
    const int begin = (a.mode == BA_MODE_FULL || fin) ? seq_start : start;
    t.delta[b] = start - seq_start;
    t.kv_begin[b] = begin;
    if (!fin) t.cache_delta[b - s] = start - seq_start;
    if (kShared && writer) {
      seg.block_delta[b] = start - seq_start;
      seg.block_kv_begin[b] = begin;
      if (!fin) seg.cache_delta[b - s] = start - seq_start;
    }
  }
  // --- key tiles of all work items of a sequence's final block, one head chunk (cached keys packed / block by block; all
  // items, then every second one)
  if (writer) {
    int d[4] = {0, 0, 0, 0};
    for (int base = 0; base < batch; base += (int)blockDim.x) {
      const int s = base + tid;
      int v[4] = {0, 0, 0, 0}, total[4];
      if (s < batch) {
        const int fin = t.cu_final_seq[s + 1] - t.cu_final_seq[s], cached = t.cu_seq[s + 1] - t.cu_seq[s] - fin;
        const int n_items = t.cu_ftile[s + 1] - t.cu_ftile[s], own = own_tiles_sum(fin, tt);
        const int n_odd = n_items / 2, own_odd = own_tiles_sum_odd(fin, tt), packed = (cached + 127) / 128;
        const int walked = t.cache_tile_cu[t.cu_seq_block[s + 1] - s - 1] - t.cache_tile_cu[t.cu_seq_block[s] - s];
        v[0] = n_items * packed + own; v[1] = n_items * walked + own;
        v[2] = n_odd * packed + own_odd; v[3] = n_odd * walked + own_odd;
      }
      cta_exclusive_scan<4>(v, total, scan_smem);
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        if (s < batch) seg.cu_stream[k * (batch + 1) + s] = d[k] + v[k];
        d[k] += total[k];
      }
    }
    if (tid == 0) {
#pragma unroll
      for (int k = 0; k < 4; ++k) seg.cu_stream[k * (batch + 1) + batch] = d[k];
      seg.totals[7] = BA_TABLES_VALID;  // kernels that walk the tables check this word first
    }
  }
  __syncthreads();
  return true;
}

// theta_m = base^(-2m/d) = 2^(m * (-2/d) * log2(base)) of the rotary pair m this thread always meets: the number of threads is
// a multiple of the pairs of a head.
__device__ __forceinline__ double thread_theta(const SegmentArgs &a) {
  return exp2((double)((blockIdx.x * blockDim.x + threadIdx.x) % a.half_dim) * a.neg2_over_d_log2_base);
}

// Everything that has one entry per token, work item or rotary pair; the grid shares it out.
__device__ __forceinline__ void segment_rows(const SegmentArgs &a, const BlockTables &t, double theta) {
  const ba_segments &seg = a.seg;
  const int batch = a.batch, B = a.B, tt = a.tile_tok;
  const int step = gridDim.x * blockDim.x, at = blockIdx.x * blockDim.x + threadIdx.x;
  float2 *rope = reinterpret_cast<float2 *>(seg.cache_rope);
  const int n_rope = (B - batch) * a.half_dim;
  for (int i = at; i < n_rope; i += step) {
    double s, co;
    sincos((double)t.cache_delta[i / a.half_dim] * theta, &s, &co);
    rope[i] = make_float2((float)co, (float)s);
  }
  for (int i = at; i < a.T; i += step) {
    const int b = upper_bound(t.cu_block, B + 1, i) - 1;
    const int local = i - t.cu_block[b];
    seg.tok_block[i] = b;
    seg.tok_pos_local[i] = local;
    seg.tok_pos[i] = t.delta[b] + local;
  }
  // work items, 32 bytes each: first query row, query rows, first own key row, first cached row, cached rows, first cached
  // block, its first key tile and the sequence's key tiles when the cached keys are walked block by block
  int4 *items = reinterpret_cast<int4 *>(seg.prompt_items);
  const int n_final = t.cu_ftile[batch], n_other = t.cu_qtile[B] - n_final;
  for (int i = at; i < n_other + n_final; i += step) {
    const int b = upper_bound(t.cu_qtile, B + 1, i) - 1, k = i - t.cu_qtile[b];
    const int s = upper_bound(t.cu_seq_block, batch + 1, b) - 1;
    const bool fin = b == t.cu_seq_block[s + 1] - 1;
    const int q0 = t.cu_block[b] + k * tt;
    // final blocks last, the others closed up (cu_ftile[s] items of final blocks come before block b)
    const int j = fin ? n_other + t.cu_ftile[s] + k : i - t.cu_ftile[s];
    items[2 * j] = make_int4(q0, min(tt, t.cu_block[b + 1] - q0), t.kv_begin[b], 0);
    items[2 * j + 1] = make_int4(0, fin ? t.cu_final_seq[s] + k * tt : 0, 0, 0);
  }
  for (int i = at; i < t.cache_tile_cu[B - batch]; i += step) seg.cache_tile_block[i] = upper_bound(t.cache_tile_cu, B - batch + 1, i) - 1;
  items = reinterpret_cast<int4 *>(seg.final_items);
  for (int i = at; i < t.cu_ftile[batch]; i += step) {
    const int s = upper_bound(t.cu_ftile, batch + 1, i) - 1;
    const int f0 = t.cu_final_seq[s], f1 = t.cu_final_seq[s + 1];
    const int q0 = f0 + (i - t.cu_ftile[s]) * tt, cached0 = t.cu_seq[s] - f0;
    const int cb0 = t.cu_seq_block[s] - s, cb1 = t.cu_seq_block[s + 1] - s - 1, tile0 = t.cache_tile_cu[cb0];
    items[2 * i] = make_int4(q0, min(tt, f1 - q0), f0, cached0);
    items[2 * i + 1] = make_int4(t.cu_seq[s + 1] - f1 - cached0, cb0, tile0, t.cache_tile_cu[cb1] - tile0);
  }
}

// Lengths passed as kernel arguments: n_blocks block lengths, then the blocks of every sequence.
template <int N>
struct InlineLengths { int32_t v[N]; };

// One launch.  kInline = 0: the lengths are device arrays.
template <int kInline, int kThreads>
__global__ void __launch_bounds__(kThreads)
ba_segment_kernel(const SegmentArgs a, const int32_t *__restrict__ lens, const int32_t *__restrict__ seq_nblocks,
                  const __grid_constant__ InlineLengths<(kInline > 0 ? kInline : 1)> in) {
  __shared__ int32_t tab[10][kThreads + 1];
  __shared__ int scan_smem[6 * 33];
  __shared__ int bad;
  __shared__ int32_t in_smem[kInline > 0 ? kInline : 1];
  if (kInline > 0) {
    for (int i = threadIdx.x; i < a.B + a.batch; i += kThreads) in_smem[i] = in.v[i];
    lens = in_smem; seq_nblocks = in_smem + a.B;
    __syncthreads();
  }
  const double theta = thread_theta(a);                  // (independent of the lengths: in front of the scans)
  ba_pdl_wait();
  ba_pdl_trigger();
  const BlockTables t = {tab[0], tab[1], tab[2], tab[3], tab[4], tab[5], tab[6], tab[7], tab[8], tab[9]};
  if (!segment_blocks<true>(a, lens, seq_nblocks, t, blockIdx.x == 0, scan_smem, &bad)) {
    if (blockIdx.x == 0 && threadIdx.x == 0) ba_record_status(a.status, BA_ERR_INVALID_ARG);
    return;
  }
  segment_rows(a, t, theta);
}

__device__ __forceinline__ BlockTables global_tables(const ba_segments &g) {
  return {g.cu_seq_block, g.cu_block, g.cu_qtile, g.block_kv_begin, g.block_delta, g.cache_tile_cu, g.cache_delta,
          g.cu_seq, g.cu_final_seq, g.cu_ftile};
}

__global__ void __launch_bounds__(1024)
ba_segment_blocks_kernel(const SegmentArgs a, const int32_t *__restrict__ lens, const int32_t *__restrict__ seq_nblocks) {
  __shared__ int scan_smem[6 * 33];
  __shared__ int bad;
  if (!segment_blocks<false>(a, lens, seq_nblocks, global_tables(a.seg), true, scan_smem, &bad) && threadIdx.x == 0)
    ba_record_status(a.status, BA_ERR_INVALID_ARG);
}

__global__ void __launch_bounds__(256) ba_segment_rows_kernel(const SegmentArgs a) {
  if (a.seg.totals[7] != BA_TABLES_VALID) return;
  segment_rows(a, global_tables(a.seg), thread_theta(a));
}

template <int N, int kThreads>
void launch_inline(const SegmentArgs &a, const int32_t *lens, const int32_t *nb, unsigned grid, cudaStream_t stream) {
  InlineLengths<N> in;
  for (int i = 0; i < a.B; ++i) in.v[i] = lens[i];
  for (int i = 0; i < a.batch; ++i) in.v[a.B + i] = nb[i];
  ba_launch(ba_segment_kernel<N, kThreads>, dim3(grid), kThreads, 0, stream, true, a, nullptr, nullptr, in);
}

}  // namespace

// block_lens / seq_nblocks: device arrays, or host arrays when `inline_lengths` (at most BA_SEGMENT_INLINE values).
ba_status ba_segment_launch(ba_ctx *ctx, const int32_t *block_lens, const int32_t *seq_nblocks, bool inline_lengths,
                            int32_t batch, int32_t n_blocks, int32_t n_tokens, int mode, int32_t gen,
                            const ba_segments *seg, cudaStream_t stream) {
  SegmentArgs a;
  a.batch = batch; a.B = n_blocks; a.T = n_tokens; a.mode = mode; a.tile_tok = seg->q_tile_tokens; a.gen = gen;
  a.half_dim = ctx->cfg.head_dim / 2;
  a.neg2_over_d_log2_base = -2.0 / (double)ctx->cfg.head_dim * log2(ctx->cfg.rope_theta);
  a.seg = *seg; a.status = ctx->dev_status;
  if (n_blocks <= kSharedBlocks) {
    // one fp64 rotation costs about as much as eight token entries
    const long long work = (long long)n_tokens + 8LL * (n_blocks - batch) * a.half_dim;
    const int threads = n_blocks <= 256 ? 256 : 1024;
    const long long want = (work + 4 * threads - 1) / (4 * threads);
    const unsigned grid = (unsigned)(want < ctx->sm_count ? want : ctx->sm_count);
    if (!inline_lengths) ba_segment_kernel<0, 1024><<<grid, 1024, 0, stream>>>(a, block_lens, seq_nblocks, InlineLengths<1>());
    else if (n_blocks + batch <= 128) launch_inline<128, 256>(a, block_lens, seq_nblocks, grid, stream);
    else if (n_blocks <= 256) launch_inline<512, 256>(a, block_lens, seq_nblocks, grid, stream);
    else launch_inline<BA_SEGMENT_INLINE, 1024>(a, block_lens, seq_nblocks, grid, stream);
    BA_CUDA_TRY(cudaGetLastError());
    ctx->launches += 1;
    return BA_OK;
  }
  ba_segment_blocks_kernel<<<1, 1024, 0, stream>>>(a, block_lens, seq_nblocks);
  BA_CUDA_TRY(cudaGetLastError());
  ba_segment_rows_kernel<<<(unsigned)((n_tokens + 255) / 256), 256, 0, stream>>>(a);
  BA_CUDA_TRY(cudaGetLastError());
  ctx->launches += 2;
  return BA_OK;
}
