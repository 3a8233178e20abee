// Internal declarations shared by the translation units of the library.
#pragma once

#include <cuda_runtime.h>
#include <cuda_bf16.h>
#include <stdint.h>
#include <stddef.h>

#include "ba.h"
#include "ba_plan.h"

// A failed runtime call also leaves its code in the runtime's per-thread "last error" slot; it is
// cleared here so that a later, healthy launch does not trip over it.
#define BA_CUDA_TRY(expr)                                              \
  do {                                                                 \
    cudaError_t _e = (expr);                                           \
    if (_e != cudaSuccess) { cudaGetLastError(); return BA_ERR_CUDA; } \
  } while (0)

// Programmatic dependent launch.  A call is a chain of short kernels (tables, re-encode, attention, merge), and between two
// of them the GPU idles for 1-2 us (a 32-layer retrieval prompt, 96 kernels: 1010 -> 897 us; forward and backward of three small
// prompts: 91 -> 66 us).  Kernels launched with ba_launch may be scheduled as soon as every CTA of the kernel
// before them in the stream has said ba_pdl_trigger() or exited: their set-up runs beside that kernel's tail.
//  * ba_pdl_wait() returns when the kernel before has completed and its writes are visible; every thread calls it before it
//    touches global memory, on every path to an exit, so that a kernel's completion implies that of all before it.  (The dQ
//    kernel of the backward pass reads beside its predecessor: it acquires a word that one released, and waits at its exit.)
//  * A kernel that allocates tensor memory triggers after its allocation: a CTA of the next kernel on the same SM must
//    never hold columns that a CTA of this one still waits for.
// A kernel launched in the ordinary way, before or after, behaves as usual.
__device__ __forceinline__ void ba_pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void ba_pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
template <class... P, class... A>
static inline cudaError_t ba_launch_clusters(void (*kernel)(P...), int cluster, dim3 grid, unsigned threads, size_t smem,
                                             cudaStream_t stream, bool early, A &&...args) {
  cudaLaunchAttribute attr[2];
  int n = 0;
  if (early) {
    attr[n].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[n++].val.programmaticStreamSerializationAllowed = 1;
  }
  if (cluster > 1) {
    attr[n].id = cudaLaunchAttributeClusterDimension;
    attr[n].val.clusterDim.x = (unsigned)cluster; attr[n].val.clusterDim.y = 1; attr[n++].val.clusterDim.z = 1;
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid; cfg.blockDim = dim3(threads); cfg.dynamicSmemBytes = smem; cfg.stream = stream;
  cfg.attrs = attr; cfg.numAttrs = (unsigned)n;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}
template <class... P, class... A>
static inline cudaError_t ba_launch(void (*kernel)(P...), dim3 grid, unsigned threads, size_t smem, cudaStream_t stream, bool early,
                                    A &&...args) {
  return ba_launch_clusters(kernel, 1, grid, threads, smem, stream, early, static_cast<A &&>(args)...);
}

// Value of ba_segments::totals[7] once ba_segment's kernel has found the lengths consistent.
#define BA_TABLES_VALID 0x600D

// One re-encoding job: block c of `n_blocks` is read from row src_off[c] (or cu[c]) of `src`,
// rotated by delta[c] with the (cos, sin) pairs in `table`, and written to rows cu[c].. of `dst`.
struct ba_reencode_job {
  const uint4 *src;
  uint4 *dst;
  const int32_t *src_off;
  const int32_t *cu;
  const int32_t *delta;
  const float2 *table;      // [n_blocks][head_dim / 2] (cos, sin)
  int32_t n_src_rows, n_blocks, n_rows;
  int32_t head_dim, row_vecs /* uint4 per row */, layout;
  // non-null: the totals of the ba_segment() tables that `cu`, `delta` or `table` belong to.  They must be valid -- of tables
  // whose lengths did not add up nothing but the totals is written -- and, with stamp != 0 (`table` is the rotation table
  // stored with them), still those of the call that stamped them; else the job reports BA_ERR_INVALID_ARG and moves nothing.
  const int32_t *totals;
  int32_t stamp;
  // non-null: the source is a paged pool -- block c owns pages page_idx[page_cu[c] .. page_cu[c+1]) of
  // 1 << page_lg rows each (src_off is ignored)
  const int32_t *page_cu, *page_idx;
  int32_t page_lg;
  // a row whose source lies outside `src`: skipped and reported (BA_ROWS_SKIPPED), or written as zeros, as an attention call
  // that reads it in place would see it
  int32_t outside;
};
constexpr int32_t BA_ROWS_SKIPPED = 0, BA_ROWS_ZERO = 1, BA_ROWS_ZERO_REPORTED = 2;

// Source row of row `t` (0-based inside its block) of a job's block `c`; negative when its page list has no good entry for it.
__device__ __forceinline__ long long ba_job_source_row(const ba_reencode_job &job, int c, int c_begin, int t) {
  if (job.page_cu) {
    const int page0 = __ldg(job.page_cu + c), k = t >> job.page_lg;
    const int page = k >= 0 && k < __ldg(job.page_cu + c + 1) - page0 ? __ldg(job.page_idx + page0 + k) : -1;
    if (page < 0) return -1;
    return ((long long)page << job.page_lg) + (t & ((1 << job.page_lg) - 1));
  }
  return (job.src_off ? (long long)__ldg(job.src_off + c) : (long long)c_begin) + t;
}

__device__ __forceinline__ bool ba_job_tables_hold(const ba_reencode_job &job) {
  if (!job.totals) return true;
  const int2 w = __ldg(reinterpret_cast<const int2 *>(job.totals + 6));    // stamp, validity (the totals are 16-byte aligned)
  return w.y == BA_TABLES_VALID && (job.stamp == 0 || w.x == job.stamp);
}

// Context: configuration, workspace and the device status word.
struct ba_ctx {
  ba_config cfg;
  int device;
  int sm_count;
  float scale;              // softmax scale actually used
  void *workspace;          // device
  size_t workspace_bytes;
  int32_t *dev_status;      // device word: first non-zero ba_status recorded by a kernel
  int64_t launches;
  int32_t last_attend[4];          // layout of the last attention launch: CTAs, partial slots, balanced tails, tail tiles
  // a re-encoding job queued by ba_reencode_k_deferred: carried along by the next attention
  // launch (or run by ba_flush); its angle table sits at the very end of the workspace
  ba_reencode_job pending;
  int has_pending;
  size_t pending_table_bytes;
  cudaStream_t pending_stream;
  // rotation table of the cached blocks built by the last ba_segment (in the caller's table buffer):
  // a re-encoding call whose delta array is that table's cache_delta reuses it instead of rebuilding it
  const int32_t *seg_delta;
  const float2 *seg_rope;
  int32_t seg_rope_blocks;
  const int32_t *seg_totals;   // totals of the same ba_segment, which stamped them with seg_stamp ([6])
  int32_t seg_stamp;
  int32_t seg_counter;      // ba_segment calls so far on this context
  // tensor maps of recently used tensors (attention launches re-use a handful of buffers)
  struct ba_map_cache *maps;
};

static inline size_t ba_align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

// Workspace layout: [0, 64 KiB) staging of host-side length arrays (ba_segment);
// [64 KiB, ...) per-call scratch: split-KV partial results (attention) or, at the very end
// of the workspace, the angle table (re-encode).  Calls on one context are stream-ordered,
// so the regions may be reused from call to call.
static inline size_t ba_scratch_offset(const ba_ctx *) { return 64 * 1024; }
// The last 256 bytes below the scratch area: three words of launch counters (attention) and, 128 bytes on, a word of the
// backward pass.
static inline int32_t *ba_counters(const ba_ctx *ctx) { return (int32_t *)((char *)ctx->workspace + ba_scratch_offset(ctx) - 256); }
static inline int32_t *ba_backward_flag(const ba_ctx *ctx) { return ba_counters(ctx) + 32; }

// Records the first device-side problem; later ones are dropped.
__device__ __forceinline__ void ba_record_status(int32_t *status, int32_t code) {
  atomicCAS(status, 0, code);
}

// Entry points implemented in the individual .cu files.
constexpr int BA_SEGMENT_INLINE = 960;    // host-side lengths passed as kernel arguments, up to this many values
ba_status ba_segment_launch(ba_ctx *ctx, const int32_t *block_lens, const int32_t *seq_nblocks, bool inline_lengths,
                            int32_t batch, int32_t n_blocks, int32_t n_tokens, int mode, int32_t gen,
                            const ba_segments *seg, cudaStream_t stream);

// Re-encoding in two steps: angle table, then the rotation itself.
ba_status ba_reencode_table_launch(ba_ctx *ctx, const int32_t *delta, int32_t n_blocks, float2 *table,
                                   cudaStream_t stream);
ba_status ba_reencode_main_launch(ba_ctx *ctx, const ba_reencode_job &job, cudaStream_t stream);
// Units of a row (a thread moves one: a 16-byte vector, or a pair of them in the half layout).  The re-encoding kernel takes
// rows of up to kBaReencodeMaxUnits: 4096 elements, 8192 in the half layout.
constexpr int kBaReencodeMaxUnits = 512;
static inline int ba_reencode_units(int layout, int row_vecs) { return layout == BA_ROPE_ADJACENT ? row_vecs : row_vecs / 2; }
ba_status ba_reencode_launch(ba_ctx *ctx, const void *k_src, const int32_t *src_off,
                             int32_t n_src_rows, void *k_dst, const int32_t *cu,
                             const int32_t *delta, int32_t n_blocks, int32_t n_rows, float2 *table,
                             cudaStream_t stream);
ba_reencode_job ba_make_reencode_job(const ba_ctx *ctx, const void *k_src, const int32_t *src_off,
                                     int32_t n_src_rows, void *k_dst, const int32_t *cu, const int32_t *delta,
                                     int32_t n_blocks, int32_t n_rows, const float2 *table);
// Runs a pending deferred job as a stand-alone launch (no-op when nothing is pending).
ba_status ba_flush_pending(ba_ctx *ctx, cudaStream_t stream);

struct ba_attend_args {
  // queries / outputs: rows of the q packing (prompt packing for prefill, final packing for final attend)
  const __nv_bfloat16 *q;
  void *o;
  float *lse;
  int32_t n_q_rows;
  int out_f32;
  // primary keys/values: same packing as q (prefill: the whole prompt; final attend: the final blocks)
  const __nv_bfloat16 *k, *v;
  int32_t n_kv_rows;
  // cached keys/values (final attend only)
  const __nv_bfloat16 *k_cache, *v_cache;
  int32_t n_cache_rows, n_v_rows;
  const int32_t *v_src_off;
  // fused warm path: k_cache holds the cached keys at cache-time positions (n_k_rows rows; block c
  // at row k_src_off[c], or at its packed offset when k_src_off is null)
  int fused;
  const int32_t *k_src_off;
  int32_t n_k_rows;
  void *k_out;     // fused call: non-null -> the re-encoded keys are written here (cache packing)
  // paged pool (page_rows > 0): the cached values -- and on the fused path the cached keys -- are read
  // through a page table instead of v_src_off / k_src_off
  int32_t page_rows;
  const int32_t *page_cu, *page_idx;
  int final_only;  // 1: ba_final_attend, 0: ba_block_prefill
  int mode;        // ba_mode
  size_t reserved_bytes;   // of the end of the workspace, in use during this call
};

ba_status ba_attend_launch(ba_ctx *ctx, const ba_attend_args &a, const ba_segments *seg,
                           cudaStream_t stream);
