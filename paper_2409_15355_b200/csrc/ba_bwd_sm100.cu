// Backward pass of attention under the Block-attention mask for sm_100a (Section 2.4: block
// fine-tuning trains with this mask in place of the lower-triangular one, so the gradients flow
// through the same masked softmax as ba_block_prefill).
//
// With P = softmax(scale Q K^T + mask), O = P V and delta_i = dO_i . O_i:
//     dV = P^T dO,   dP = dO V^T,   dS = P * (dP - delta),   dQ = scale dS K,   dK = scale dS^T Q.
// P is recomputed from the log-sum-exp the forward pass stored.  Two kernels, both built from
// 128 x 128 tiles on the tensor cores (tcgen05.mma, accumulators in tensor memory), neither uses
// atomics, so results are run-to-run identical:
//   * ba_bwd_dkv_kernel: one CTA owns 128 keys of one block and one KV head and walks over every
//     query tile that sees them (all heads of the group).  It forms the scores transposed, S^T = K Q^T
//     and dP^T = V dO^T (keys on the tensor-memory lanes, query rows on the columns), so that its
//     threads -- two per key -- write P^T and dS^T back to tensor memory as bf16, where they are the A
//     operands of dV += P^T dO and dK += dS^T Q (nothing goes through shared memory, nothing is transposed).
//   * ba_bwd_dq_kernel: one CTA owns one query tile (tokens x heads of one KV group, as in the
//     forward kernel) and walks over the key tiles it sees: S = Q K^T, dP = dO V^T (query rows on the
//     lanes), dS written to tensor memory, dQ += dS K.
// The tiles a CTA walks over (Q and dO there, K and V here) are double-buffered in shared memory, so the
// loads of the next tile run under the current one.
//
// Both are bound by the chain scores -> threads -> gradient products rather than by the tensor core alone, so both are
// laid out to keep the tensor core busy while threads work: the dK/dV kernel hands P^T over before it touches dP^T, so that
// dV and the next tile's S^T run under the formation of dS^T, and dK and the next dP^T under the next P^T; the dQ kernel
// runs two CTAs per SM.  The dK/dV score products take 128 columns at a time: a 64-column product reads as much of its A
// operand from shared memory as a 128-column one.  8 x 16384 ragged tokens, 32/8 heads of 128, one B200: dK/dV 6.49 -> 5.28 ms, dQ
// 6.04 -> 4.15 ms against kernels that worked in steps of 64 columns with one CTA per SM.
#include <math.h>
#include <type_traits>

#include "ba_common.cuh"
#include "ba_sm100.cuh"

using namespace sm100;

int ba_heads_per_tile(const ba_config &c);

namespace {

// dK/dV kernel: eight row warps, two threads per key (tensor-memory lane), each with one half of a tile's 128 query
// rows; warp 8 issues the products, warp 9 the loads.
constexpr int kDkvThreads = 320;
constexpr int kDkvMmaWarp = 8, kDkvLoadWarp = 9;
// dQ kernel: one group of four row warps, a product warp and a load warp; two CTAs share an SM.
constexpr int kDqThreads = 192;
constexpr int kDqMmaWarp = 4, kDqLoadWarp = 5;
constexpr int kTile = 128;
constexpr int kStep = 64;              // keys a step of the dQ kernel works on

struct BwdParams {
  const float *lse;          // [T, Hq] natural-log softmax denominators of the forward pass
  const float *delta;        // [T, Hq] dO . O
  int32_t *started;          // 0 until the dK/dV kernel of this call has seen all that was written before it; then 1 + the query
                             // tile pairs of the tables, or -1 when they are not valid
  void *dq, *dk, *dv;
  int out_f32;
  int32_t *status;
  int Hq, Hkv, G, hpt, hpt_log2, tok;
  float scale, scale_log2;
  int mode;
  int n_rows;                // T
  ba_segments seg;
};

// Shared memory of the dK/dV kernel: K and V tiles that stay, two buffers of (Q, dO) tiles it walks over, and what
// every key has to know about a query row -- -lse * log2 e, -dO . O * scale, visible keys of the tile --, two buffers of each.
template <int D>
struct DkvLayout {
  static constexpr int kChunks = D / 64;
  static constexpr int kRegion = 128 * 128;              // 128 rows x 128 bytes
  static constexpr int kTileBytes = 128 * D * 2;
  static constexpr int kFix0 = 0, kFix1 = kTileBytes;
  static constexpr int kWalk = 2 * kTileBytes;            // buffer b: tiles at kWalk + b * 2 * kTileBytes, + kTileBytes
  static constexpr int kStats = 6 * kTileBytes;           // [buffer][3][128]
  static constexpr int kCtrl = kStats + 2 * 3 * 128 * 4;
  static constexpr int kBytes = kCtrl + 256;
};

struct DkvCtrl {
  uint64_t fix_full, walk_full[2], walk_free[2];
  uint64_t s_full, dp_full;              // S^T / dP^T of the tile are in tensor memory
  uint64_t p_done, ds_done;              // P^T / dS^T of the tile are in tensor memory
  uint64_t fin;                          // every product of the CTA has completed
  uint32_t tmem_base;
  int abort_flag;
};

// Shared memory of the dQ kernel: Q and dO tiles that stay, two 64-key tiles of K and one of V.  At head_dim 128 this is
// 112 KB + 1 KB: exactly half of what an SM has for two CTAs, so the base must be 1024-byte aligned as it is.
template <int D>
struct DqLayout {
  static constexpr int kChunks = D / 64;
  static constexpr int kRegion = 128 * 128;
  static constexpr int kTileBytes = 128 * D * 2;
  static constexpr int kKeyRegion = kStep * 128;          // 64 rows x 128 bytes
  static constexpr int kKeyBytes = kStep * D * 2;
  static constexpr int kQ = 0, kDo = kTileBytes;
  static constexpr int kK = 2 * kTileBytes;               // K of step i at kK + (i & 1) * kKeyBytes
  static constexpr int kV = kK + 2 * kKeyBytes;
  static constexpr int kCtrl = kV + kKeyBytes;
  static constexpr int kBytes = kCtrl + 1024;
};

struct DqCtrl {
  uint64_t fix_full, k_full[2], k_free[2], v_full, v_free;
  uint64_t sd_full;                      // S and dP of the step are in tensor memory
  uint64_t s_read;                       // the row threads hold S in registers: the next step's S may overwrite it
  uint64_t rows_done;                    // dS of the step is in tensor memory
  uint64_t fin;
  uint32_t tmem_base;
  int abort_flag;
};

__device__ __forceinline__ void tmem_st16(uint32_t taddr, const uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], "
      "{%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16};"
      ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]),
        "r"(r[8]), "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15])
      : "memory");
}
__device__ __forceinline__ void row_warps_barrier() { asm volatile("bar.sync 1, 256;" ::: "memory"); }

// The i < n with a[i] <= x < a[i + 1], for ascending a with a[0] <= x < a[n]; by a warp, 32 places at a time (each round is one
// latency of L2, and a CTA waits for it before it can ask for its first tile; a binary search over 130 blocks takes eight.  With the
// look-ups behind the request for K and V: 8 x 16384 ragged tokens, forward and backward, 13464 -> 13410 us).
__device__ __forceinline__ int warp_find(const int32_t *a, int n, int x) {
  int lo = 0, hi = n;
  while (hi - lo > 1) {
    const int step = (hi - lo + 31) / 32, i = lo + (int)(threadIdx.x & 31) * step;
    const unsigned below = __ballot_sync(0xffffffffu, i < hi && __ldg(a + i) <= x);
    lo += (31 - __clz((int)below)) * step;
    hi = min(hi, lo + step);
  }
  return lo;
}
// The dQ kernel reads what other kernels wrote behind an acquire, not behind a wait: with ordinary loads, as the read-only path
// (which the compiler may also take by itself) need not see it.
template <class T>
__device__ __forceinline__ T ld_plain(const T *p) {
  static_assert(sizeof(T) == 4, "one word");
  uint32_t v;
  asm volatile("ld.global.b32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return *reinterpret_cast<T *>(&v);
}
// BwdParams::started, once it is not zero; 0 when that takes a second (it is set before the kernel that asks can start).
__device__ __forceinline__ int32_t wait_started(const int32_t *started) {
  int32_t v = ld_acquire(started);
  if (v == 0) {
    const unsigned long long t0 = global_ns();
    while ((v = ld_acquire(started)) == 0 && global_ns() - t0 <= kWaitLimitNs) __nanosleep(kSleepNs);
  }
  return v;
}

__device__ __forceinline__ uint64_t mul2(uint64_t a, uint64_t b) {
  uint64_t d;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ uint32_t bf16_pair(float lo, float hi) {
  __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<uint32_t *>(&v);
}

// The arithmetic of these helpers is packed fp32x2: for a pair of columns, x = s * scale_log2 - lse_log2 (one FMA),
// p = exp2(x) (two), t = dp * scale - delta * scale (one FMA), ds = p * t (one multiply).  kMasked = false is for
// steps in which every (row, key) pair is visible: no comparison at all.
//
// dQ kernel, one query row (= lane) against 32 keys: dS as bf16, two per register.  Keys 0 .. n_ok - 1 are visible.
template <bool kMasked>
__device__ __forceinline__ void bwd_row_ds(const uint32_t *s, const uint32_t *dp, uint32_t (&dw)[16], int n_ok, float scale_log2,
                                           float neg_lse_log2, float neg_delta_scaled, float scale) {
  const uint64_t sl2 = pack2(scale_log2, scale_log2), nl2 = pack2(neg_lse_log2, neg_lse_log2);
  const uint64_t sc2 = pack2(scale, scale), nd2 = pack2(neg_delta_scaled, neg_delta_scaled);
#pragma unroll
  for (int i = 0; i < 16; ++i) {
    const uint64_t x2 = fma2(pack2(__uint_as_float(s[2 * i]), __uint_as_float(s[2 * i + 1])), sl2, nl2);
    float x0, x1;
    unpack2(x2, x0, x1);
    float p0 = ex2(x0), p1 = ex2(x1);
    if (kMasked) {
      if (2 * i >= n_ok) p0 = 0.f;
      if (2 * i + 1 >= n_ok) p1 = 0.f;
    }
    const uint64_t t2 = fma2(pack2(__uint_as_float(dp[2 * i]), __uint_as_float(dp[2 * i + 1])), sc2, nd2);
    float d0, d1;
    unpack2(mul2(pack2(p0, p1), t2), d0, d1);
    dw[i] = bf16_pair(d0, d1);
  }
}

// dK/dV kernel, one key (= lane `j`) against 32 query rows (= columns).  The per-row values come from shared memory,
// the same address for every thread; lim = number of keys of this tile the row sees.  First P^T: fp32 in place of s
// (the second half of the step needs it), bf16 in pw.
template <bool kMasked>
__device__ __forceinline__ void dkv_p(uint32_t *s, uint32_t (&pw)[16], int j, const float *neg_lse2, const int *lim, float scale_log2) {
  const uint64_t sl2 = pack2(scale_log2, scale_log2);
#pragma unroll
  for (int q = 0; q < 8; ++q) {                          // four columns at a time: one 16-byte read of each per-row array
    const ulonglong2 l4 = *reinterpret_cast<const ulonglong2 *>(neg_lse2 + 4 * q);
    int4 m4 = make_int4(0, 0, 0, 0);
    if (kMasked) m4 = *reinterpret_cast<const int4 *>(lim + 4 * q);
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      const int i = 2 * q + e;
      const uint64_t x2 = fma2(pack2(__uint_as_float(s[2 * i]), __uint_as_float(s[2 * i + 1])), sl2, e ? l4.y : l4.x);
      float x0, x1;
      unpack2(x2, x0, x1);
      float p0 = ex2(x0), p1 = ex2(x1);
      if (kMasked) {
        if (j >= (e ? m4.z : m4.x)) p0 = 0.f;
        if (j >= (e ? m4.w : m4.y)) p1 = 0.f;
      }
      s[2 * i] = __float_as_uint(p0); s[2 * i + 1] = __float_as_uint(p1);
      pw[i] = bf16_pair(p0, p1);
    }
  }
}
// Then dS^T = P^T (dP^T - dO . O) scale.
__device__ __forceinline__ void dkv_ds(const uint32_t *p, const uint32_t *dp, uint32_t (&dw)[16], const float *neg_dls, float scale) {
  const uint64_t sc2 = pack2(scale, scale);
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    const ulonglong2 d4 = *reinterpret_cast<const ulonglong2 *>(neg_dls + 4 * q);
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      const int i = 2 * q + e;
      const uint64_t t2 = fma2(pack2(__uint_as_float(dp[2 * i]), __uint_as_float(dp[2 * i + 1])), sc2, e ? d4.y : d4.x);
      float d0, d1;
      unpack2(mul2(pack2(__uint_as_float(p[2 * i]), __uint_as_float(p[2 * i + 1])), t2), d0, d1);
      dw[i] = bf16_pair(d0, d1);
    }
  }
}

// Writes the first n_rows of a warp's 32 accumulator rows (D fp32 columns of tensor memory, lane = row) to global memory.  row_at(r):
// element offset of row r in dst.  The rows go through shared memory (`stage`: 32 rows of 2 D bytes, 16-byte chunk c of row r at
// chunk position c ^ (r & 7)), so that a store instruction writes whole bf16 rows or halves of fp32 rows, 2 D bytes in a run: 16
// bytes each of 32 rows fill no sector.  The loops stay loops: the code is passed once, and fetching it costs more than running it.
// (8 x 16384 ragged tokens, forward and backward: 13580 -> 13464 us; three small prompts 63.8 -> 63.0.)  Only rows that exist are
// gone through: blocks of 1-20 tokens leave most of a tile's rows empty (2 x 8192 tokens of them: 1582 us with stores from the
// threads' own rows, 1634 with all 32 rows passed, 1572; 4/4 heads, blocks of 50-500: 389, 393, 382).
template <int D, class RowAt>
__device__ __forceinline__ void store_acc_rows(uint32_t tAcc, uint8_t *stage, void *dst, int out_f32, int n_rows, RowAt row_at) {
  constexpr int kRowBytes = 2 * D, kChunks = kRowBytes / 16;
  if (n_rows <= 0) return;
  const int lane = threadIdx.x & 31, c = lane % kChunks;
  uint8_t *own = stage + lane * kRowBytes;
#pragma unroll 1
  for (int h = 0; h < (out_f32 ? 2 : 1); ++h) {            // kRowBytes of every row at a time
#pragma unroll 1
    for (int k = 0; k < (out_f32 ? D / 64 : D / 32); ++k) {
      uint32_t a[32];
      tmem_ld_32x32b_x32(tAcc + h * (D / 2) + k * 32, a);
      tmem_wait_ld();
      if (out_f32) {
#pragma unroll
        for (int i = 0; i < 8; ++i)
          *reinterpret_cast<uint4 *>(own + (((k * 8 + i) ^ (lane & 7)) << 4)) = make_uint4(a[4 * i], a[4 * i + 1], a[4 * i + 2], a[4 * i + 3]);
      } else {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          uint32_t w[4];
#pragma unroll
          for (int e = 0; e < 4; ++e) w[e] = bf16_pair(__uint_as_float(a[8 * i + 2 * e]), __uint_as_float(a[8 * i + 2 * e + 1]));
          *reinterpret_cast<uint4 *>(own + (((k * 4 + i) ^ (lane & 7)) << 4)) = make_uint4(w[0], w[1], w[2], w[3]);
        }
      }
    }
    __syncwarp();
#pragma unroll 4
    for (int r = lane / kChunks; r < n_rows; r += 32 / kChunks) {
      const uint4 x = *reinterpret_cast<const uint4 *>(stage + r * kRowBytes + ((c ^ (r & 7)) << 4));
      *reinterpret_cast<uint4 *>(reinterpret_cast<uint8_t *>(dst) + row_at(r) * (out_f32 ? 4 : 2) + h * kRowBytes + c * 16) = x;
    }
    __syncwarp();
  }
}

// ---------------------------------------------------------------------------------------------
// dK, dV: CTA = (128-key tile of one block, KV head)
// ---------------------------------------------------------------------------------------------
template <int D>
__global__ void __launch_bounds__(kDkvThreads, 1)
ba_bwd_dkv_kernel(const __grid_constant__ CUtensorMap tmap_q, const __grid_constant__ CUtensorMap tmap_do,
                  const __grid_constant__ CUtensorMap tmap_k, const __grid_constant__ CUtensorMap tmap_v,
                  const BwdParams p) {
  using L = DkvLayout<D>;
  extern __shared__ uint8_t smem_raw[];
  uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  DkvCtrl *ctrl = reinterpret_cast<DkvCtrl *>(smem + L::kCtrl);
  const int tid = threadIdx.x, warp = tid >> 5;
  const ba_segments &sg = p.seg;
  ba_pdl_wait();
  if (blockIdx.x == gridDim.x - 1) {                       // a CTA without keys: off the way of those the dQ kernel waits for
    if (tid == 0 && blockIdx.y == 0) st_release(p.started, __ldg(sg.totals + 7) == BA_TABLES_VALID ? __ldg(sg.totals + 2) + 1 : -1);
    return;
  }
  const int valid = __ldg(sg.totals + 7), n_ktiles = __ldg(sg.cu_ktile + sg.n_blocks);
  // which keys: tile `kt` of the batch (a tile never spans two blocks), KV head `g`
  const int kt = blockIdx.x, g = blockIdx.y;
  if (valid != BA_TABLES_VALID || kt >= n_ktiles) return;
  const int b = warp_find(sg.cu_ktile, sg.n_blocks, kt);
  const int blk0 = __ldg(sg.cu_block + b), blk1 = __ldg(sg.cu_block + b + 1);
  const int k0 = blk0 + (kt - __ldg(sg.cu_ktile + b)) * kTile;
  const int n_keys = min(kTile, blk1 - k0);
  if (tid == 0) {
    mbar_init(&ctrl->fix_full, 1); mbar_init(&ctrl->fin, 1);
    for (int i = 0; i < 2; ++i) { mbar_init(&ctrl->walk_full[i], 1); mbar_init(&ctrl->walk_free[i], 1); }
    mbar_init(&ctrl->s_full, 1); mbar_init(&ctrl->dp_full, 1);
    mbar_init(&ctrl->p_done, 256); mbar_init(&ctrl->ds_done, 256);
    ctrl->abort_flag = 0;
    fence_barrier_init();
  }
  if (warp == kDkvMmaWarp) { tmem_alloc(&ctrl->tmem_base, 512); tmem_relinquish(); }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = ctrl->tmem_base;
  volatile int *abort_flag = &ctrl->abort_flag;
  ba_pdl_trigger();
  const uint32_t tST = tmem, tDPT = tmem + 128, tDV = tmem + 256, tDK = tmem + 384;

  if (warp == kDkvLoadWarp && elect_one()) {               // (before the look-ups that follow)
    mbar_arrive_expect_tx(&ctrl->fix_full, 2 * L::kTileBytes);
    for (int c = 0; c < L::kChunks; ++c) {
      tma_load_3d(smem + L::kFix0 + c * L::kRegion, &tmap_k, &ctrl->fix_full, c * 64, g, k0);
      tma_load_3d(smem + L::kFix1 + c * L::kRegion, &tmap_v, &ctrl->fix_full, c * 64, g, k0);
    }
  }
  // which queries see them: rows k0 .. end of the block (causally); in full mode the rest of the sequence
  // as well; in block mode the rows of the sequence's final block (they see every earlier block)
  const int sq = __ldg(sg.block_seq + b);
  const int seq1 = __ldg(sg.cu_seq + sq + 1);
  const int fin0 = __ldg(sg.cu_block + __ldg(sg.cu_seq_block + sq + 1) - 1);    // first row of the final block
  const bool is_final = __ldg(sg.block_is_final + b) != 0;
  const int r1_begin = k0, r1_end = (p.mode == BA_MODE_FULL) ? seq1 : blk1;     // causal range
  int r2_begin = 0, r2_end = 0;                                                 // range that sees all the keys
  if (p.mode == BA_MODE_BLOCK && !is_final) { r2_begin = fin0; r2_end = seq1; }
  const int tiles1 = (r1_end - r1_begin + p.tok - 1) / p.tok, tiles2 = (r2_end - r2_begin + p.tok - 1) / p.tok;
  const int n_chunks = p.G / p.hpt;                                             // head chunks of this KV group
  const int n_iter = (tiles1 + tiles2) * n_chunks;
  // iteration `it`: token tile it / n_chunks, head chunk it % n_chunks
  auto iter_rows = [&](int it, int &row0, int &row_end, bool &causal, int &head0) {
    const int ti = it / n_chunks, ch = it - ti * n_chunks;
    causal = ti < tiles1;
    row0 = causal ? r1_begin + ti * p.tok : r2_begin + (ti - tiles1) * p.tok;
    row_end = causal ? r1_end : r2_end;
    head0 = g * p.G + ch * p.hpt;
  };

  if (warp == kDkvLoadWarp) {
    if (elect_one()) {
      bool ok = true;
      int it = 0;
      for (; it < n_iter; ++it) {                        // Q and dO tiles of tile `it` into buffer it & 1
        ok = mbar_wait(&ctrl->walk_free[it & 1], ((it >> 1) & 1) ^ 1, abort_flag);
        if (!ok) break;
        int row0, row_end, head0; bool causal;
        iter_rows(it, row0, row_end, causal, head0);
        uint8_t *dst = smem + L::kWalk + (it & 1) * 2 * L::kTileBytes;
        mbar_arrive_expect_tx(&ctrl->walk_full[it & 1], 2 * L::kTileBytes);
        for (int c = 0; c < L::kChunks; ++c) {
          tma_load_3d(dst + c * L::kRegion, &tmap_q, &ctrl->walk_full[it & 1], c * 64, head0, row0);
          tma_load_3d(dst + L::kTileBytes + c * L::kRegion, &tmap_do, &ctrl->walk_full[it & 1], c * 64, head0, row0);
        }
      }
      if (!ok) {                                         // leave no copy in flight: wait (bounded) for those already requested
        for (uint32_t spin = 0; spin < (1u << 20) && !mbar_try_wait(&ctrl->fix_full, 0); ++spin) { }
        for (int k = max(0, it - 2); k < it; ++k)
          for (uint32_t spin = 0; spin < (1u << 20) && !mbar_try_wait(&ctrl->walk_full[k & 1], (k >> 1) & 1); ++spin) { }
      }
    }
  } else if (warp == kDkvMmaWarp) {
    if (elect_one()) {
      constexpr uint32_t idesc_nt = make_idesc_bf16(128, kTile, 0);             // both operands K-major
      constexpr uint32_t idesc_tn = make_idesc_bf16(128, D, 1);                 // A from tensor memory, B MN-major
      const uint64_t k_desc = make_smem_desc(smem_u32(smem + L::kFix0), 16, 1024);
      const uint64_t v_desc = make_smem_desc(smem_u32(smem + L::kFix1), 16, 1024);
      // scores of the tile in walk buffer `buf`: S^T = K Q^T (which = 0) or dP^T = V dO^T (1)
      auto issue_scores = [&](int buf, int which) {
        const uint64_t a_desc = which ? v_desc : k_desc;
        const uint64_t b_desc = make_smem_desc(smem_u32(smem + L::kWalk + (buf * 2 + which) * L::kTileBytes), 16, 1024);
#pragma unroll
        for (int k = 0; k < D / 16; ++k) {
          const uint64_t off = (uint64_t)(((k >> 2) * L::kRegion + (k & 3) * 32) >> 4);
          mma_ss(which ? tDPT : tST, a_desc + off, b_desc + off, idesc_nt, k > 0);
        }
        mma_commit(which ? &ctrl->dp_full : &ctrl->s_full);
      };
      // gradients: dV += P^T dO (which = 0) or dK += dS^T Q (1), 16 query rows at a time
      auto issue_grads = [&](int buf, int which, bool first) {
        const uint64_t b_mn = make_smem_desc(smem_u32(smem + L::kWalk + (buf * 2 + (which ^ 1)) * L::kTileBytes), L::kRegion, 1024);
#pragma unroll
        for (int k = 0; k < 8; ++k)
          mma_ts(which ? tDK : tDV, (which ? tDPT : tST) + (k >> 2) * 64 + (k & 3) * 8, b_mn + (uint64_t)((k * 16 * 128) >> 4), idesc_tn,
                 (!first || k > 0) ? 1u : 0u);
      };
      bool ok = mbar_wait(&ctrl->fix_full, 0, abort_flag);
      if (ok && n_iter > 0) ok = mbar_wait(&ctrl->walk_full[0], 0, abort_flag);
      if (ok && n_iter > 0) { tc_fence_after(); issue_scores(0, 0); issue_scores(0, 1); }
      for (int it = 0; it < n_iter && ok; ++it) {
        const int buf = it & 1;
        const bool more = it + 1 < n_iter;
        // the next tile's S^T follows dV on the tensor pipe (P^T has been read then) and runs while the threads form dS^T;
        // its dP^T follows dK and runs while they form the next P^T
        ok = mbar_wait(&ctrl->p_done, it & 1, abort_flag);
        if (!ok) break;
        tc_fence_after();
        issue_grads(buf, 0, it == 0);
        if (more) {
          ok = mbar_wait(&ctrl->walk_full[buf ^ 1], ((it + 1) >> 1) & 1, abort_flag);
          if (!ok) break;
          tc_fence_after();
          issue_scores(buf ^ 1, 0);
        }
        ok = mbar_wait(&ctrl->ds_done, it & 1, abort_flag);
        if (!ok) break;
        tc_fence_after();
        issue_grads(buf, 1, it == 0);
        mma_commit(&ctrl->walk_free[buf]);
        if (more) issue_scores(buf ^ 1, 1);
      }
      if (ok) mma_commit(&ctrl->fin);
    }
  } else {
    const int j = tid & 127;                             // key of the tile = tensor-memory lane
    const int h = warp >> 2;                             // this thread's half of every tile: query rows 64 h .. + 63
    const uint32_t lane_off = (uint32_t)((warp & 3) * 32) << 16;
    float *stats = reinterpret_cast<float *>(smem + L::kStats);
    // thread tid < 128 fetches what the keys need to know about query row `tid`, one tile ahead
    float n_lse = 0.f, n_dls = 0.f; int n_lim = 0;
    auto fetch_stats = [&](int it) {
      int row0, row_end, head0; bool causal;
      iter_rows(it, row0, row_end, causal, head0);
      const int tok_i = row0 + (tid >> p.hpt_log2);
      const int head = head0 + (tid & (p.hpt - 1));
      n_lse = 0.f; n_dls = 0.f; n_lim = 0;
      if (tok_i < row_end) {
        n_lse = __ldg(p.lse + (size_t)tok_i * p.Hq + head);                    // (used a tile later: nothing waits for them here)
        n_dls = __ldg(p.delta + (size_t)tok_i * p.Hq + head);
        n_lim = causal ? max(0, min(n_keys, tok_i - k0 + 1)) : n_keys;         // keys 0 .. n_lim - 1 of the tile are visible
      }
    };
    if (tid < 128 && n_iter > 0) fetch_stats(0);
    bool ok = true;
    int it = 0;
    for (; it < n_iter; ++it) {
      float *st = stats + (it & 1) * 3 * 128;
      if (tid < 128) {
        st[tid] = n_lse * -1.4426950408889634f; st[128 + tid] = -n_dls * p.scale; reinterpret_cast<int *>(st)[256 + tid] = n_lim;
        if (it + 1 < n_iter) fetch_stats(it + 1);
      }
      row_warps_barrier();
      int row0, row_end, head0; bool causal;
      iter_rows(it, row0, row_end, causal, head0);
      // every pair of this thread's half visible?  (all 128 keys exist, the rows exist and, in the causal range,
      // already the first one sees the tile's last key)
      const int tok_first = row0 + ((h * 64) >> p.hpt_log2), tok_last = row0 + ((h * 64 + 63) >> p.hpt_log2);
      const bool all_visible = n_keys == kTile && tok_last < row_end && (!causal || tok_first - k0 + 1 >= kTile);
      const uint32_t a = tST + h * 64 + lane_off, d = tDPT + h * 64 + lane_off;
      const float *lse = st + h * 64, *dls = st + 128 + h * 64;
      const int *lim = reinterpret_cast<const int *>(st) + 256 + h * 64;
      uint32_t s[64], w[16];
      ok = mbar_wait(&ctrl->s_full, it & 1, abort_flag);
      if (!ok) break;
      tc_fence_after();
      // P^T as bf16 over the S^T columns the thread has read, two per column: the A operand of dV
      auto form_p = [&](auto masked) {
        constexpr bool kMasked = decltype(masked)::value;
        tmem_ld_32x32b_x32(a, *reinterpret_cast<uint32_t(*)[32]>(&s[0]));
        tmem_wait_ld();
        tmem_ld_32x32b_x32(a + 32, *reinterpret_cast<uint32_t(*)[32]>(&s[32]));
        dkv_p<kMasked>(s, w, j, lse, lim, p.scale_log2);
        tmem_st16(a, w);
        tmem_wait_ld();
        dkv_p<kMasked>(s + 32, w, j, lse + 32, lim + 32, p.scale_log2);
        tmem_st16(a + 16, w);
        tmem_wait_st();
      };
      if (all_visible) form_p(std::false_type{});
      else form_p(std::true_type{});
      tc_fence_before();
      mbar_arrive(&ctrl->p_done);
      ok = mbar_wait(&ctrl->dp_full, it & 1, abort_flag);
      if (!ok) break;
      tc_fence_after();
      uint32_t d0[32], d1[32];
      tmem_ld_32x32b_x32(d, d0);
      tmem_wait_ld();
      tmem_ld_32x32b_x32(d + 32, d1);
      dkv_ds(s, d0, w, dls, p.scale);
      tmem_st16(d, w);
      tmem_wait_ld();
      dkv_ds(s + 32, d1, w, dls + 32, p.scale);
      tmem_st16(d + 16, w);
      tmem_wait_st();
      tc_fence_before();
      mbar_arrive(&ctrl->ds_done);
    }
    // a warp that gave up a wait still comes to the barriers the others may be on their way to: those have no limit
    __syncwarp();
    for (++it; it < n_iter; ++it) row_warps_barrier();
    // accumulators: lane = key row of the tile; one thread of a key writes dV, the other dK
    if (ok && n_iter > 0) ok = mbar_wait(&ctrl->fin, 0, abort_flag);
    if (ok && n_iter > 0) {
      tc_fence_after();
      const int j0 = (warp & 3) * 32;
      store_acc_rows<D>((h ? tDK : tDV) + lane_off, smem + (h ? L::kFix1 : L::kFix0) + j0 * (2 * D), h ? p.dk : p.dv, p.out_f32, min(32, n_keys - j0),
                        [&](int r) { return ((size_t)(k0 + j0 + r) * p.Hkv + g) * D; });
    }
  }
  tc_fence_before();
  __syncthreads();
  if (tid == 0 && ctrl->abort_flag) ba_record_status(p.status, BA_ERR_TIMEOUT);
  if (warp == kDkvMmaWarp) tmem_dealloc(tmem, 512);
}

// ---------------------------------------------------------------------------------------------
// dQ: CTA = (query tile of `tok` tokens x `hpt` heads, head chunk)
// ---------------------------------------------------------------------------------------------
// Two CTAs share an SM (half of the shared memory and 256 of the 512 tensor-memory columns each): while the threads of
// one turn scores into dS, the tensor core works for the other, and one's start-up and write-out hide under the
// other's products.
template <int D>
__global__ void __launch_bounds__(kDqThreads, 2)
ba_bwd_dq_kernel(const __grid_constant__ CUtensorMap tmap_q, const __grid_constant__ CUtensorMap tmap_do,
                 const __grid_constant__ CUtensorMap tmap_k, const __grid_constant__ CUtensorMap tmap_v,
                 const BwdParams p, int n_tiles_upper, int n_head_chunks) {
  using L = DqLayout<D>;
  extern __shared__ __align__(1024) uint8_t smem_dq[];
  uint8_t *smem = smem_dq;
  DqCtrl *ctrl = reinterpret_cast<DqCtrl *>(smem + L::kCtrl);
  const int tid = threadIdx.x, warp = tid >> 5;
  const ba_segments &sg = p.seg;
  // This kernel needs nothing of the dK/dV kernel but what that one had to wait for itself (dO . O, the tables, the inputs): it
  // starts on the SMs that one leaves (unless dq takes the place of an input) and waits for it only before it ends.  Until then
  // nothing makes the earlier kernels' writes visible here but the word that the dK/dV kernel released after its own wait, so
  // every thread acquires it first (the copy engine's reads: behind a proxy fence).
  struct WaitAtExit { __device__ ~WaitAtExit() { ba_pdl_wait(); } } wait_at_exit;
  const int32_t n_pairs_1 = wait_started(p.started);
  if (n_pairs_1 == 0) ba_record_status(p.status, BA_ERR_TIMEOUT);

  // query tile: one half of a query-tile pair of the forward kernel, an item of ba_segment's list (one line of it: behind the
  // acquire nothing is in L1).  Tiles are taken from the end of the list (final blocks, then within a sequence the last ones: those
  // see the most keys), all head chunks of a tile side by side.
  const int qt = n_tiles_upper - 1 - (int)blockIdx.x / n_head_chunks;
  const int pair = qt >> 1, half = qt & 1;
  if (pair + 1 >= n_pairs_1) return;                      // (no tables, or no such pair)
  const int32_t *item = sg.prompt_items + 8 * (size_t)pair;
  const int row0 = ld_plain(item), n_rows = ld_plain(item + 1), kv0 = ld_plain(item + 2);   // row i sees keys kv0 .. i
  const int q0 = row0 + half * p.tok;
  if (q0 >= row0 + n_rows) return;
  const int q_end = min(q0 + p.tok, row0 + n_rows);       // rows q0 .. q_end - 1
  const int head0 = ((int)blockIdx.x % n_head_chunks) * p.hpt, g = head0 / p.G;
  const int n_steps = (q_end - kv0 + kStep - 1) / kStep;  // step i: keys kv0 + 64 i .. + 63

  if (tid == 0) {
    mbar_init(&ctrl->fix_full, 1); mbar_init(&ctrl->fin, 1);
    for (int i = 0; i < 2; ++i) { mbar_init(&ctrl->k_full[i], 1); mbar_init(&ctrl->k_free[i], 1); }
    mbar_init(&ctrl->v_full, 1); mbar_init(&ctrl->v_free, 1);
    mbar_init(&ctrl->sd_full, 1); mbar_init(&ctrl->s_read, 128); mbar_init(&ctrl->rows_done, 128);
    ctrl->abort_flag = 0;
    fence_barrier_init();
  }
  if (warp == kDqMmaWarp) { tmem_alloc(&ctrl->tmem_base, 256); tmem_relinquish(); }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = ctrl->tmem_base;
  volatile int *abort_flag = &ctrl->abort_flag;
  ba_pdl_trigger();
  const uint32_t tS = tmem, tDP = tmem + 64, tDQ = tmem + 128;   // S and dP of one step (64 keys each), dQ

  if (warp == kDqLoadWarp) {
    if (elect_one()) {
      fence_proxy_async_global();
      mbar_arrive_expect_tx(&ctrl->fix_full, 2 * L::kTileBytes);
      for (int c = 0; c < L::kChunks; ++c) {
        tma_load_3d(smem + L::kQ + c * L::kRegion, &tmap_q, &ctrl->fix_full, c * 64, head0, q0);
        tma_load_3d(smem + L::kDo + c * L::kRegion, &tmap_do, &ctrl->fix_full, c * 64, head0, q0);
      }
      bool ok = true;
      int nk = 0, nv = 0;                                // tiles of K and V requested so far
      for (int i = 0; i < n_steps; ++i) {
        ok = mbar_wait(&ctrl->k_free[i & 1], ((i >> 1) & 1) ^ 1, abort_flag);
        if (!ok) break;
        mbar_arrive_expect_tx(&ctrl->k_full[i & 1], L::kKeyBytes);
        for (int c = 0; c < L::kChunks; ++c)
          tma_load_3d(smem + L::kK + (i & 1) * L::kKeyBytes + c * L::kKeyRegion, &tmap_k, &ctrl->k_full[i & 1], c * 64, g, kv0 + i * kStep);
        ++nk;
        ok = mbar_wait(&ctrl->v_free, (i & 1) ^ 1, abort_flag);
        if (!ok) break;
        mbar_arrive_expect_tx(&ctrl->v_full, L::kKeyBytes);
        for (int c = 0; c < L::kChunks; ++c)
          tma_load_3d(smem + L::kV + c * L::kKeyRegion, &tmap_v, &ctrl->v_full, c * 64, g, kv0 + i * kStep);
        ++nv;
      }
      if (!ok) {                                         // leave no copy in flight: wait (bounded) for those already requested
        for (uint32_t spin = 0; spin < (1u << 20) && !mbar_try_wait(&ctrl->fix_full, 0); ++spin) { }
        for (int k = max(0, nk - 2); k < nk; ++k)
          for (uint32_t spin = 0; spin < (1u << 20) && !mbar_try_wait(&ctrl->k_full[k & 1], (k >> 1) & 1); ++spin) { }
        if (nv > 0)
          for (uint32_t spin = 0; spin < (1u << 20) && !mbar_try_wait(&ctrl->v_full, (nv - 1) & 1); ++spin) { }
      }
    }
  } else if (warp == kDqMmaWarp) {
    if (elect_one()) {
      constexpr uint32_t idesc_nt = make_idesc_bf16(128, kStep, 0);
      constexpr uint32_t idesc_nn = make_idesc_bf16(128, D, 1);                 // A from tensor memory (dS), B MN-major (K)
      const uint64_t q_desc = make_smem_desc(smem_u32(smem + L::kQ), 16, 1024);
      const uint64_t do_desc = make_smem_desc(smem_u32(smem + L::kDo), 16, 1024);
      const uint64_t v_desc = make_smem_desc(smem_u32(smem + L::kV), 16, 1024);
      auto issue_s = [&](int i) -> bool {                // S = Q K^T for the 64 keys of step i
        if (!mbar_wait(&ctrl->k_full[i & 1], (i >> 1) & 1, abort_flag)) return false;
        tc_fence_after();
        const uint64_t k_desc = make_smem_desc(smem_u32(smem + L::kK + (i & 1) * L::kKeyBytes), 16, 1024);
#pragma unroll
        for (int k = 0; k < D / 16; ++k) {
          const uint64_t qo = (uint64_t)(((k >> 2) * L::kRegion + (k & 3) * 32) >> 4);
          const uint64_t ko = (uint64_t)(((k >> 2) * L::kKeyRegion + (k & 3) * 32) >> 4);
          mma_ss(tS, q_desc + qo, k_desc + ko, idesc_nt, k > 0);
        }
        return true;
      };
      auto issue_dp = [&](int i) -> bool {               // dP = dO V^T
        if (!mbar_wait(&ctrl->v_full, i & 1, abort_flag)) return false;
        tc_fence_after();
#pragma unroll
        for (int k = 0; k < D / 16; ++k) {
          const uint64_t qo = (uint64_t)(((k >> 2) * L::kRegion + (k & 3) * 32) >> 4);
          const uint64_t vo = (uint64_t)(((k >> 2) * L::kKeyRegion + (k & 3) * 32) >> 4);
          mma_ss(tDP, do_desc + qo, v_desc + vo, idesc_nt, k > 0);
        }
        mma_commit(&ctrl->sd_full);
        mma_commit(&ctrl->v_free);
        return true;
      };
      bool ok = mbar_wait(&ctrl->fix_full, 0, abort_flag);
      if (ok && n_steps > 0) ok = issue_s(0) && issue_dp(0);
      for (int i = 0; i < n_steps && ok; ++i) {
        // the next step's S is formed while the threads still work on this step: they hold S in registers
        if (i + 1 < n_steps) {
          ok = mbar_wait(&ctrl->s_read, i & 1, abort_flag);
          if (!ok) break;
          tc_fence_after();
          ok = issue_s(i + 1);
          if (!ok) break;
        }
        ok = mbar_wait(&ctrl->rows_done, i & 1, abort_flag);
        if (!ok) break;
        tc_fence_after();
        const uint64_t k_mn = make_smem_desc(smem_u32(smem + L::kK + (i & 1) * L::kKeyBytes), L::kKeyRegion, 1024);
#pragma unroll
        for (int k = 0; k < kStep / 16; ++k)             // dQ += dS K, 16 keys at a time
          mma_ts(tDQ, tDP + k * 8, k_mn + (uint64_t)((k * 16 * 128) >> 4), idesc_nn, (i > 0 || k > 0) ? 1u : 0u);
        mma_commit(&ctrl->k_free[i & 1]);
        if (i + 1 < n_steps) ok = issue_dp(i + 1);       // (behind dQ on the tensor pipe: dS has been read)
      }
      if (ok) mma_commit(&ctrl->fin);
    }
  } else {
    const int r = tid;                                   // row of the query tile = tensor-memory lane
    const uint32_t lane_off = (uint32_t)(warp * 32) << 16;
    const int tok_i = q0 + (r >> p.hpt_log2);
    const int head = head0 + (r & (p.hpt - 1));
    const bool row_ok = tok_i < q_end;
    float nlse = 0.f, ndl = 0.f;
    if (row_ok) {
      nlse = ld_plain(p.lse + (size_t)tok_i * p.Hq + head) * -1.4426950408889634f;
      ndl = -ld_plain(p.delta + (size_t)tok_i * p.Hq + head) * p.scale;
    }
    bool ok = true;
    for (int i = 0; i < n_steps; ++i) {
      const int kr = kv0 + i * kStep;
      const int n_ok = row_ok ? max(0, min(kStep, tok_i - kr + 1)) : 0;
      // every pair of this step visible?  (every row of the tile exists and already the first one sees the step's last key)
      const bool all_visible = q0 + p.tok <= q_end && q0 - kr + 1 >= kStep;
      ok = mbar_wait(&ctrl->sd_full, i & 1, abort_flag);
      if (!ok) break;
      tc_fence_after();
      auto step = [&](auto masked) {
        constexpr bool kMasked = decltype(masked)::value;
        uint32_t s[64], d0[32], d1[32], dw[16];
        tmem_ld_32x32b_x32(tS + lane_off, *reinterpret_cast<uint32_t(*)[32]>(&s[0]));
        tmem_ld_32x32b_x32(tS + lane_off + 32, *reinterpret_cast<uint32_t(*)[32]>(&s[32]));
        tmem_ld_32x32b_x32(tDP + lane_off, d0);
        tmem_wait_ld();
        tc_fence_before();
        mbar_arrive(&ctrl->s_read);
        tmem_ld_32x32b_x32(tDP + lane_off + 32, d1);
        bwd_row_ds<kMasked>(s, d0, dw, n_ok, p.scale_log2, nlse, ndl, p.scale);
        tmem_st16(tDP + lane_off, dw);                   // dS as bf16 over the dP columns that have been read
        tmem_wait_ld();
        bwd_row_ds<kMasked>(s + 32, d1, dw, n_ok - 32, p.scale_log2, nlse, ndl, p.scale);
        tmem_st16(tDP + lane_off + 16, dw);
        tmem_wait_st();
      };
      if (all_visible) step(std::false_type{});
      else step(std::true_type{});
      tc_fence_before();
      mbar_arrive(&ctrl->rows_done);
    }
    if (ok && n_steps > 0) ok = mbar_wait(&ctrl->fin, 0, abort_flag);
    if (ok && n_steps > 0) {
      tc_fence_after();
      store_acc_rows<D>(tDQ + lane_off, smem + L::kQ + warp * 32 * (2 * D), p.dq, p.out_f32, min(32, ((q_end - q0) << p.hpt_log2) - warp * 32),
                        [&](int i) {
        const int row = warp * 32 + i, tk = q0 + (row >> p.hpt_log2);
        return ((size_t)tk * p.Hq + head0 + (row & (p.hpt - 1))) * D;
      });
    }
  }
  tc_fence_before();
  __syncthreads();
  if (tid == 0 && ctrl->abort_flag) ba_record_status(p.status, BA_ERR_TIMEOUT);
  if (warp == kDqMmaWarp) tmem_dealloc(tmem, 256);
}

// delta[row, head] = dO . O: D / 8 threads per (row, head), each with one 16-byte vector of both operands
template <int D>
__global__ void __launch_bounds__(256)
ba_bwd_delta_kernel(const __nv_bfloat16 *__restrict__ o, const __nv_bfloat16 *__restrict__ d_o, float *__restrict__ delta,
                    int n_rows_heads, int32_t *started) {
  ba_pdl_wait();
  ba_pdl_trigger();
  if (blockIdx.x == 0 && threadIdx.x == 0) *started = 0;
  constexpr int kLanes = D / 8;                          // 8 or 16 threads per row
  const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  const long long rh = t / kLanes;
  const int v = (int)(t - rh * kLanes);
  float acc = 0.f;
  if (rh < n_rows_heads) {
    const uint4 a = __ldg(reinterpret_cast<const uint4 *>(o + rh * D) + v);
    const uint4 b = __ldg(reinterpret_cast<const uint4 *>(d_o + rh * D) + v);
    const uint32_t aw[4] = {a.x, a.y, a.z, a.w}, bw[4] = {b.x, b.y, b.z, b.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      acc = fmaf(__uint_as_float(aw[i] << 16), __uint_as_float(bw[i] << 16), acc);
      acc = fmaf(__uint_as_float(aw[i] & 0xffff0000u), __uint_as_float(bw[i] & 0xffff0000u), acc);
    }
  }
#pragma unroll
  for (int sft = kLanes / 2; sft > 0; sft >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, sft);
  if (rh < n_rows_heads && v == 0) delta[rh] = acc;
}

typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                  const cuuint64_t *, const cuuint32_t *, const cuuint32_t *,
                                  CUtensorMapInterleave, CUtensorMapSwizzle, CUtensorMapL2promotion,
                                  CUtensorMapFloatOOBfill);

bool bwd_make_map(CUtensorMap *m, const void *ptr, int D, int heads, long long rows, int box_heads, int box_rows) {
  static EncodeTiledFn enc = nullptr;
  if (!enc) {
    void *fp = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &fp, cudaEnableDefault, &q) != cudaSuccess) return false;
    enc = reinterpret_cast<EncodeTiledFn>(fp);
  }
  if (!enc || rows < 1) return false;
  cuuint64_t dims[3] = {(cuuint64_t)D, (cuuint64_t)heads, (cuuint64_t)rows};
  cuuint64_t strides[2] = {(cuuint64_t)D * 2, (cuuint64_t)heads * D * 2};
  cuuint32_t box[3] = {64, (cuuint32_t)box_heads, (cuuint32_t)box_rows};
  cuuint32_t es[3] = {1, 1, 1};
  return enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void *>(ptr), dims, strides, box, es,
             CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
             CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

bool overlap(const void *a, size_t a_bytes, const void *b, size_t b_bytes) {
  const uintptr_t x = (uintptr_t)a, y = (uintptr_t)b;
  return x < y + b_bytes && y < x + a_bytes;
}

// dq_in_place: dq takes the place of q or d_o.  A CTA of the dQ kernel has its own rows of both in shared memory before it writes
// them, but the dK/dV kernel reads all of them: the dQ kernel must not start before that one has ended.
template <int D>
ba_status launch_bwd(ba_ctx *ctx, const BwdParams &p, bool dq_in_place, const CUtensorMap &tq, const CUtensorMap &tdo, const CUtensorMap &tk,
                     const CUtensorMap &tv, const CUtensorMap &tk64, const CUtensorMap &tv64, int n_ktiles_upper, int n_pairs_upper,
                     cudaStream_t stream) {
  BA_CUDA_TRY(ba_launch(ba_bwd_dkv_kernel<D>, dim3((unsigned)n_ktiles_upper + 1, (unsigned)p.Hkv), kDkvThreads, DkvLayout<D>::kBytes + 1024,
                        stream, true, tq, tdo, tk, tv, p));
  const int n_head_chunks = p.Hq / p.hpt;
  BA_CUDA_TRY(ba_launch(ba_bwd_dq_kernel<D>, dim3((unsigned)(2 * n_pairs_upper) * n_head_chunks), kDqThreads, DqLayout<D>::kBytes, stream,
                        !dq_in_place, tq, tdo, tk64, tv64, p, 2 * n_pairs_upper, n_head_chunks));
  ctx->launches += 2;
  return BA_OK;
}

}  // namespace

// Per-context set-up (device current): the kernels' shared-memory limit is raised once.
ba_status ba_bwd_sm100_setup(ba_ctx *) {
  BA_CUDA_TRY(cudaFuncSetAttribute(ba_bwd_dkv_kernel<128>, cudaFuncAttributeMaxDynamicSharedMemorySize, DkvLayout<128>::kBytes + 1024));
  BA_CUDA_TRY(cudaFuncSetAttribute(ba_bwd_dq_kernel<128>, cudaFuncAttributeMaxDynamicSharedMemorySize, DqLayout<128>::kBytes));
  BA_CUDA_TRY(cudaFuncSetAttribute(ba_bwd_dkv_kernel<64>, cudaFuncAttributeMaxDynamicSharedMemorySize, DkvLayout<64>::kBytes + 1024));
  BA_CUDA_TRY(cudaFuncSetAttribute(ba_bwd_dq_kernel<64>, cudaFuncAttributeMaxDynamicSharedMemorySize, DqLayout<64>::kBytes));
  return BA_OK;
}

ba_status ba_bwd_sm100_launch(ba_ctx *ctx, const void *q, const void *k, const void *v, const void *o,
                              const float *lse, const void *d_o, void *dq, void *dk, void *dv, int out_f32,
                              const ba_segments *seg, int mode, cudaStream_t stream) {
  const int D = ctx->cfg.head_dim, Hq = ctx->cfg.n_q_heads, Hkv = ctx->cfg.n_kv_heads;
  const int T = seg->n_tokens;
  BwdParams p;
  p.lse = lse; p.dq = dq; p.dk = dk; p.dv = dv; p.out_f32 = out_f32; p.status = ctx->dev_status;
  p.Hq = Hq; p.Hkv = Hkv; p.G = Hq / Hkv;
  p.hpt = ba_heads_per_tile(ctx->cfg);
  p.hpt_log2 = p.hpt == 4 ? 2 : p.hpt == 2 ? 1 : 0;
  p.tok = 128 / p.hpt;
  p.scale = ctx->scale;
  p.scale_log2 = ctx->scale * 1.4426950408889634f;
  p.mode = mode; p.n_rows = T; p.seg = *seg;
  if (seg->q_tile_tokens != 2 * p.tok || !seg->cu_ktile || !seg->prompt_items) return BA_ERR_INVALID_ARG;
  // delta = dO . O sits in the scratch area of the workspace
  const size_t need = (size_t)T * Hq * sizeof(float);
  if (!ctx->workspace || ctx->workspace_bytes < ba_scratch_offset(ctx) + need) return BA_ERR_WORKSPACE;
  float *delta = reinterpret_cast<float *>(reinterpret_cast<char *>(ctx->workspace) + ba_scratch_offset(ctx));
  p.delta = delta;
  p.started = ba_backward_flag(ctx);
  const int n_rh = T * Hq;
  const long long threads = (long long)n_rh * (D / 8);
  BA_CUDA_TRY(ba_launch(D == 128 ? ba_bwd_delta_kernel<128> : ba_bwd_delta_kernel<64>, dim3((unsigned)((threads + 255) / 256)), 256, 0,
                        stream, true, (const __nv_bfloat16 *)o, (const __nv_bfloat16 *)d_o, delta, n_rh, p.started));
  ctx->launches += 1;
  CUtensorMap tq, tdo, tk, tv, tk64, tv64;
  if (!bwd_make_map(&tq, q, D, Hq, T, p.hpt, p.tok) || !bwd_make_map(&tdo, d_o, D, Hq, T, p.hpt, p.tok) ||
      !bwd_make_map(&tk, k, D, Hkv, T, 1, kTile) || !bwd_make_map(&tv, v, D, Hkv, T, 1, kTile) ||
      !bwd_make_map(&tk64, k, D, Hkv, T, 1, kStep) || !bwd_make_map(&tv64, v, D, Hkv, T, 1, kStep))
    return BA_ERR_CUDA;
  const int n_ktiles_upper = T / kTile + seg->n_blocks;
  const int n_pairs_upper = seg->n_prompt_items > 0 ? seg->n_prompt_items : T / (2 * p.tok) + seg->n_blocks;
  const size_t q_bytes = (size_t)T * Hq * D * 2, dq_bytes = out_f32 ? 2 * q_bytes : q_bytes;
  const bool dq_in_place = overlap(dq, dq_bytes, q, q_bytes) || overlap(dq, dq_bytes, d_o, q_bytes);
  if (D == 128) return launch_bwd<128>(ctx, p, dq_in_place, tq, tdo, tk, tv, tk64, tv64, n_ktiles_upper, n_pairs_upper, stream);
  return launch_bwd<64>(ctx, p, dq_in_place, tq, tdo, tk, tv, tk64, tv64, n_ktiles_upper, n_pairs_upper, stream);
}
