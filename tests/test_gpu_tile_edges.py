"""Kernels and launch variants at the sizes where they can go wrong -- tile edges, remainders, the smallest and the
largest of a range -- against the fp64 oracle.  Tolerances are those of the parity tests: outputs max-abs 1e-2 /
mean-abs 1e-3 (fp32 stores), gradients relative Frobenius 1e-2 (P and dS are rounded to bf16 before the products)."""
import numpy as np
import pytest
import torch

from oracle import block_attention as ob
from paper_2409_15355_b200 import binding as B
from paper_2409_15355_b200 import runtime as R
from paper_2409_15355_b200 import workloads as W
from tests.test_gpu_backward import check_grad, run_forward_backward
from tests.test_gpu_parity import check_attention, check_reencoded, run_prefill, run_warm

pytestmark = pytest.mark.gpu

# Block lengths around the 64-key step of the dQ kernel, the 128-key tile of the dK/dV kernel and one / several query tiles.
EDGE_BLOCKS = {"steps": [1, 63, 64, 65], "tiles": [127, 128, 129, 2], "long_last": [64, 257, 191], "short_last": [320, 129, 1]}


@pytest.mark.parametrize("lens", EDGE_BLOCKS.values(), ids=EDGE_BLOCKS.keys())
@pytest.mark.parametrize("heads", [(8, 2, 128), (6, 2, 64), (2, 2, 128)], ids=str)
def test_backward_tile_edges(lens, heads):
    w = W.Workload("edges", *heads, 1e4, lens + lens[::-1], [len(lens)] * 2, seed=81)
    for mode in (B.BA_MODE_BLOCK, B.BA_MODE_FULL):
        dq, dk, dv, q, k, v, g = run_forward_backward(w, mode)
        rq, rk, rv = ob.block_prefill_backward(q, k, v, g, w.block_lens, w.seq_nblocks, mode)
        check_grad("dq", dq, rq); check_grad("dk", dk, rk); check_grad("dv", dv, rv)

# Gradients leave as whole rows of the tiles' rows that exist: blocks that end in any of a warp's rows, next to rows of other blocks
@pytest.mark.parametrize("heads", [(8, 2, 128), (6, 2, 64), (2, 2, 128)], ids=str)
@pytest.mark.parametrize("dtype", [B.BA_OUT_F32, B.BA_OUT_BF16], ids=["f32", "bf16"])
def test_backward_row_counts(heads, dtype):
    lens = [1, 2, 3, 4, 5, 7, 8, 9, 15, 17, 31, 32, 33, 34, 36, 95, 97, 1]
    w = W.Workload("row_counts", *heads, 1e4, lens + lens[::-1], [len(lens)] * 2, seed=83)
    dq, dk, dv, q, k, v, g = run_forward_backward(w, B.BA_MODE_BLOCK, grad_dtype=dtype)
    rq, rk, rv = ob.block_prefill_backward(q, k, v, g, w.block_lens, w.seq_nblocks, B.BA_MODE_BLOCK)
    check_grad("dq", dq, rq); check_grad("dk", dk, rk); check_grad("dv", dv, rv)      # (a row not written is NaN)


# The search for a key tile's block, 32 places a round: one round, two, three; gradients stored as bf16 and fp32 rows.
@pytest.mark.parametrize("n_blocks", [31, 32, 33, 1024, 1025])
@pytest.mark.parametrize("dtype", [B.BA_OUT_F32, B.BA_OUT_BF16], ids=["f32", "bf16"])
def test_backward_many_blocks(n_blocks, dtype):
    lens = [1 + i * 7 % 4 for i in range(n_blocks)]
    lens[0] = lens[-1] = 130
    w = W.Workload("many_blocks", 2, 1, 64, 1e4, lens, [n_blocks // 8] * 8 + ([n_blocks % 8] if n_blocks % 8 else []), seed=82)
    dq, dk, dv, q, k, v, g = run_forward_backward(w, B.BA_MODE_BLOCK, grad_dtype=dtype)
    rq, rk, rv = ob.block_prefill_backward(q, k, v, g, w.block_lens, w.seq_nblocks, B.BA_MODE_BLOCK)
    check_grad("dq", dq, rq); check_grad("dk", dk, rk); check_grad("dv", dv, rv)


def _ragged_lens(n_blocks, seed):
    return [int(v) for v in np.random.default_rng(seed).integers(1, 9, n_blocks)]


# ba_segment: one launch with the lengths as kernel arguments (two sizes of them), one launch from a staged copy, two launches
@pytest.mark.parametrize("n_blocks,batch", [(1, 1), (127, 1), (126, 2), (127, 2), (256, 256), (257, 3), (955, 5), (956, 5), (1024, 7), (1025, 7), (1500, 1100)])
def test_segment_launch_variants(n_blocks, batch):
    counts = [n_blocks // batch + (1 if i < n_blocks % batch else 0) for i in range(batch)]
    lens = _ragged_lens(n_blocks, n_blocks)
    lens[-1] = 700                                           # a final block of several work items
    c = R.Context(8, 2, 64, 1e4)
    tables = []
    for host in (True, False):
        a, b = np.asarray(lens, dtype=np.int32), np.asarray(counts, dtype=np.int32)
        if not host:
            a, b = torch.from_numpy(a).cuda(), torch.from_numpy(b).cuda()
        seg, buf = c.segment(a, b, B.BA_MODE_BLOCK, n_tokens=sum(lens))
        got = R.read_tables(seg, buf)
        base, raw = buf.data_ptr(), buf.cpu().numpy()
        rope = raw[seg.cache_rope - base:][:seg.n_cached_blocks * 32 * 8].view(np.float32).reshape(-1, 32, 2)
        items = raw[seg.final_items - base:][:int(got["totals"][3]) * 32].view(np.int32).reshape(-1, 8)
        stream = raw[seg.cu_stream - base:][:(batch + 1) * 16].view(np.int32).reshape(4, -1)
        tables.append((got, rope.copy(), items.copy(), stream.copy()))
    assert c.device_status() == B.BA_OK
    ref = ob.segment_tables(lens, counts, B.BA_MODE_BLOCK)
    for got, rope, items, stream in tables:
        for k in ("cu_block", "block_delta", "block_kv_begin", "cache_cu", "cache_delta", "tok_block", "tok_pos", "cu_final_seq"):
            assert got[k].tolist() == ref[k].tolist(), k
        angle = ref["cache_delta"].astype(np.float64)[:, None] * 1e4 ** (-2.0 * np.arange(32) / 64)
        assert np.abs(rope[..., 0] - np.cos(angle)).max(initial=0) < 1e-6 and np.abs(rope[..., 1] - np.sin(angle)).max(initial=0) < 1e-6
        want, sums, b0 = [], [[0], [0], [0], [0]], 0
        for s, n in enumerate(counts):
            seq = lens[b0:b0 + n]
            f0, cached0 = int(ref["cu_final_seq"][s]), int(ref["cu_seq"][s]) - int(ref["cu_final_seq"][s])
            walked, cached, per = sum(-(-v // 128) for v in seq[:-1]), sum(seq[:-1]), [0, 0, 0, 0]
            for q in range(0, seq[-1], seg.q_tile_tokens):
                rows = min(seg.q_tile_tokens, seq[-1] - q)
                want.append([f0 + q, rows, f0, cached0, cached, b0 - s, int(got["cache_tile_cu"][b0 - s]), walked])
                own = -(-(q + rows) // 128)
                odd = q // seg.q_tile_tokens % 2
                for k, tiles in enumerate((-(-cached // 128) + own, walked + own)):
                    per[k] += tiles
                    per[2 + k] += odd * tiles
            for k in range(4):
                sums[k].append(sums[k][-1] + per[k])
            b0 += n
        assert items.tolist() == want and stream.tolist() == sums
    c.close()


def _requests(name, n, seed, cached, final, heads=(8, 2, 128), pool=False):
    """n requests of cached[0] blocks of cached[1]..cached[2] tokens and a final block of final[0]..final[1]."""
    rng = np.random.default_rng(seed)
    lens, counts, pool_lens, idx = [], [], None, None
    if pool:
        pool_lens, idx = [int(v) for v in rng.integers(cached[1], cached[2] + 1, 20)], []
    for _ in range(n):
        if pool:
            idx.append([int(v) for v in rng.integers(0, 20, cached[0])])
            seq = [pool_lens[i] for i in idx[-1]]
        else:
            seq = [int(v) for v in rng.integers(cached[1], cached[2] + 1, cached[0])]
        lens += seq + [int(rng.integers(final[0], final[1] + 1))]
        counts.append(len(seq) + 1)
    return W.Workload(name, *heads, 1e4, lens, counts, seed=seed, pool_lens=pool_lens, request_pool_idx=idx)


STREAM_CASES = [_requests("more_items_than_sms", 40, 91, (4, 100, 300), (60, 200)),      # most items whole, some cut once
                _requests("fewer_items", 22, 92, (5, 1, 400), (65, 130)),                # about one piece and a half per CTA
                _requests("one_long_among_short", 45, 93, (1, 1, 2500), (64, 65)),
                _requests("two_chunks_a_group", 60, 94, (4, 90, 300), (40, 140), heads=(8, 1, 64)),
                _requests("pool", 60, 95, (5, 20, 290), (33, 129), pool=True)]


@pytest.mark.parametrize("w", STREAM_CASES, ids=lambda w: w.name)
@pytest.mark.parametrize("fused", [False, True], ids=["reencode_then_attend", "fused"])
def test_stream_launch(w, fused):
    shapes = []
    o, lse, o_ref, lse_ref = run_warm(w, B.BA_MODE_BLOCK, fused=fused, shape_out=shapes)
    assert shapes[0]["ctas"] <= 148 and shapes[0]["partials"] > 1 and shapes[0]["balanced_tails"] == 0
    check_attention(o, o_ref, lse, lse_ref)
    again = run_warm(w, B.BA_MODE_BLOCK, fused=fused)
    assert np.array_equal(o, again[0]) and np.array_equal(lse, again[1])


# The key tiles of the final blocks' items split in a prefill: one sequence and several, bf16 and fp32 stores
@pytest.mark.parametrize("w", [_requests("one", 1, 96, (9, 150, 400), (65, 65)), _requests("three", 3, 97, (7, 64, 300), (1, 200)),
                               _requests("half_head", 2, 98, (8, 100, 300), (129, 129), heads=(6, 2, 64))], ids=lambda w: w.name)
def test_prefill_with_split_final_blocks(w):
    o, lse, o_ref, lse_ref = run_prefill(w, B.BA_MODE_BLOCK)
    check_attention(o, o_ref, lse, lse_ref)
    o, lse, _, _ = run_prefill(w, B.BA_MODE_BLOCK, out_dtype=B.BA_OUT_BF16)
    check_attention(o, o_ref, lse, lse_ref, bf16_store=True)
    c = R.Context.for_workload(w)
    seg, buf = c.segment(w.block_lens, w.seq_nblocks, B.BA_MODE_BLOCK)
    x = torch.zeros(w.n_tokens, w.n_q_heads, w.head_dim, dtype=torch.bfloat16, device="cuda")
    kv = torch.zeros(w.n_tokens, w.n_kv_heads, w.head_dim, dtype=torch.bfloat16, device="cuda")
    B.ba_block_prefill(c.ctx, x, kv, kv, x, None, seg, B.BA_MODE_BLOCK, B.BA_OUT_BF16)
    assert c.last_attend_shape()["partials"] > 1
    c.close()


# bf16 rows leave as whole tiles (one copy) where a query tile is full and row by row where it is not: full, partly filled
# and missing second tiles, many entries per CTA, a background job (one pair of query buffers), 1 / 2 / 4 heads per tile
@pytest.mark.parametrize("heads", [(32, 8, 128), (8, 4, 64), (6, 2, 64)], ids=str)
@pytest.mark.parametrize("background", [False, True], ids=["plain", "background_job"])
def test_prefill_bf16_rows_full_and_ragged_tiles(heads, background):
    rng = np.random.default_rng(101)
    lens = [64, 32, 33, 1, 128, 96, 256, 65, 160] + [int(v) for v in rng.integers(1, 300, 60)]
    w = W.Workload("rows", *heads, 1e4, lens, [20, 30, 19], seed=101)
    x = [R.bits_to_device(b) for b in W.prefill_inputs(w)]
    o32 = torch.full((w.n_tokens, heads[0], heads[2]), float("nan"), dtype=torch.float32, device="cuda")
    o16 = torch.full_like(o32, float("nan"), dtype=torch.bfloat16)
    c = R.Context.for_workload(w)
    seg, buf = c.segment(w.block_lens, w.seq_nblocks, B.BA_MODE_BLOCK)
    B.ba_block_prefill(c.ctx, *x, o32, None, seg, B.BA_MODE_BLOCK, B.BA_OUT_F32)
    k_re = torch.empty(w.n_tokens - sum(w.final_lens()), heads[1], heads[2], dtype=torch.bfloat16, device="cuda")
    for _ in range(3):
        o16.fill_(float("nan"))
        if background:
            B.ba_reencode_k_deferred(c.ctx, x[1], None, w.n_tokens, k_re, seg.cache_cu, seg.cache_delta, seg.n_cached_blocks, len(k_re))
        B.ba_block_prefill(c.ctx, *x, o16, None, seg, B.BA_MODE_BLOCK, B.BA_OUT_BF16)
        assert torch.equal(o16, o32.to(torch.bfloat16))      # the same fp32 rows, rounded to nearest even
    assert c.device_status() == B.BA_OK
    c.close()


# A short final block over a cache of a few key tiles: the CTAs of a cluster share an item and merge in shared memory.
# Cluster sizes 2 .. 8, one and two query tiles per item, clusters of one query tile and of whole items, both packings of heads, CTAs that get no tile, bf16 and fp32 rows.
@pytest.mark.parametrize("w", [_requests("two_tiles", 1, 111, (1, 120, 120), (3, 3), heads=(4, 2, 64)),
                               _requests("three_tiles", 2, 112, (3, 70, 90), (33, 64), heads=(8, 2, 128)),
                               _requests("five_tiles", 3, 113, (4, 20, 200), (1, 130), heads=(8, 8, 128)),
                               _requests("ragged_sizes", 5, 114, (3, 1, 500), (1, 70), heads=(8, 1, 64)),
                               _requests("twenty_tiles", 1, 115, (9, 200, 340), (64, 64), heads=(32, 8, 128)),
                               _requests("odd_group", 2, 116, (6, 100, 300), (100, 140), heads=(6, 2, 64)),
                               _requests("one_and_two_query_tiles", 2, 117, (7, 100, 300), (65, 120), heads=(8, 2, 128))], ids=lambda w: w.name)
@pytest.mark.parametrize("fused", [False, True], ids=["reencode_then_attend", "fused"])
def test_cluster_launch(w, fused):
    shapes = []
    o, lse, o_ref, lse_ref = run_warm(w, B.BA_MODE_BLOCK, fused=fused, shape_out=shapes)
    items = sum(-(-n // (256 // _hpt(w))) for n in w.final_lens()) * (w.n_q_heads // _hpt(w))
    assert shapes[0]["partials"] == 1 and shapes[0]["ctas"] in [items * n * m for n in range(2, 9) for m in (1, 2)]
    check_attention(o, o_ref, lse, lse_ref)
    o, lse, _, _ = run_warm(w, B.BA_MODE_BLOCK, out_dtype=B.BA_OUT_BF16, fused=fused)
    check_attention(o, o_ref, lse, lse_ref, bf16_store=True)


# Items of one query tile, whose key tiles both softmax groups of a CTA share: one, two, three and more key tiles a CTA (an odd number
# leaves the groups unequal, one leaves the second idle), CTAs of a cluster with unequal numbers, a last tile used in half, values
# walked in a pool.
@pytest.mark.parametrize("w", [_requests("one_each", 1, 141, (2, 64, 100), (32, 32), heads=(8, 2, 128)),
                               _requests("ragged", 4, 142, (9, 40, 300), (1, 32), heads=(32, 8, 128)),
                               _requests("many_tiles", 4, 143, (20, 300, 400), (5, 32), heads=(32, 8, 128)),
                               _requests("narrow_heads", 6, 144, (7, 100, 400), (100, 128), heads=(6, 2, 64)),
                               _requests("pool", 3, 145, (9, 20, 290), (1, 30), heads=(8, 2, 128), pool=True)], ids=lambda w: w.name)
def test_cluster_launch_one_query_tile(w):
    shapes = []
    o, lse, o_ref, lse_ref = run_warm(w, B.BA_MODE_BLOCK, shape_out=shapes)
    items = w.n_q_heads // _hpt(w) * w.batch
    assert shapes[0]["partials"] == 1 and shapes[0]["ctas"] in [items * m for m in range(2, 9)]
    check_attention(o, o_ref, lse, lse_ref)
    again, lse_again, _, _ = run_warm(w, B.BA_MODE_BLOCK)
    assert np.array_equal(o, again) and np.array_equal(lse, lse_again)


# Rows of the longest final block, which decide whether CTAs of whole items share key tiles: counted from lengths on the host only
@pytest.mark.parametrize("w", [_requests("one", 1, 146, (2, 10, 40), (33, 33)), _requests("mixed", 4, 147, (2, 10, 40), (1, 70))], ids=lambda w: w.name)
def test_longest_final_block(w):
    c = R.Context.for_workload(w)
    seg, buf = c.segment(w.block_lens, w.seq_nblocks, B.BA_MODE_BLOCK)
    assert seg.final_rows_max == max(w.final_lens())
    lens, counts = (torch.tensor(v, dtype=torch.int32, device="cuda") for v in (w.block_lens, w.seq_nblocks))
    assert c.segment(lens, counts, B.BA_MODE_BLOCK, n_tokens=w.n_tokens)[0].final_rows_max == 0
    c.close()


def _hpt(w):
    g = w.n_q_heads // w.n_kv_heads
    return 4 if g % 4 == 0 else 2 if g % 2 == 0 else 1


# ba_reencode_k: CTAs whose rows lie in one block and CTAs that cross blocks, both rotary layouts, all sources
@pytest.mark.parametrize("layout", [B.BA_ROPE_ADJACENT, B.BA_ROPE_HALF], ids=["adjacent", "half"])
@pytest.mark.parametrize("heads", [(8, 8, 128), (2, 1, 64), (6, 3, 64)], ids=str)
def test_reencode_rows_in_one_block_and_across(layout, heads):
    lens = [1, 2, 3, 4, 5, 7, 8, 9, 31, 32, 33, 100, 1, 1, 64, 17]
    w = W.Workload("rows", *heads, 1e4, lens + [5], [len(lens) + 1], seed=121)
    c = R.Context(*heads, 1e4, rope_layout=layout)
    seg, buf = c.segment(w.block_lens, w.seq_nblocks, B.BA_MODE_BLOCK)
    t = ob.segment_tables(w.block_lens, w.seq_nblocks)
    packed = W.normal_bf16(122, (sum(lens), heads[1], heads[2]))
    want = ob.reencode_blocks(W.bf16_bits_to_f64(packed), None, t["cache_cu"], t["cache_delta"], 1e4, layout)
    src = R.bits_to_device(packed)
    out = torch.full_like(src, float("nan"))
    B.ba_reencode_k(c.ctx, src, None, len(src), out, seg.cache_cu, seg.cache_delta, len(lens), len(src))
    assert c.device_status() == B.BA_OK
    check_reencoded(R.device_to_bits(out), want)
    pool, page_cu, page_idx, n_pages = W.scatter_into_pages(packed, lens, 16, 123)
    keep = [R.bits_to_device(pool), torch.from_numpy(page_cu).cuda(), torch.from_numpy(page_idx).cuda()]
    paged = torch.full_like(src, float("nan"))
    B.ba_reencode_k_paged(c.ctx, keep[0], B.make_page_table(16, n_pages, keep[1], keep[2]), paged, seg.cache_cu, seg.cache_delta,
                          len(lens), len(src))
    assert c.device_status() == B.BA_OK and torch.equal(paged, out)
    c.close()


# The fused call over final blocks of several query tiles: in two steps through the workspace, through k_out, and (a workspace
# without room for the keys) in one
@pytest.mark.parametrize("w", [_requests("one", 1, 131, (6, 50, 300), (200, 200)), _requests("pool", 5, 132, (4, 20, 290), (70, 129), pool=True)],
                         ids=lambda w: w.name)
def test_fused_call_in_two_steps(w):
    o, lse, o_ref, lse_ref = run_warm(w, B.BA_MODE_BLOCK, fused=True)
    check_attention(o, o_ref, lse, lse_ref)
    x, t = W.warm_inputs(w), ob.segment_tables(w.block_lens, w.seq_nblocks)
    k_src, v_src = (R.bits_to_device(x[n]) for n in (("k_pool", "v_pool") if w.pool_lens else ("k_cache", "v_cache")))
    off = torch.from_numpy(x["src_off"]).cuda() if w.pool_lens else None
    q, k, v = (R.bits_to_device(x[n]) for n in ("q_f", "k_f", "v_f"))
    cfg = B.ba_config(w.n_q_heads, w.n_kv_heads, w.head_dim, 0, w.rope_theta, 0.0, 0)
    Tc, Tf = t["n_cached_tokens"], t["n_final_tokens"]
    for room in (B.ba_workspace_bytes(cfg, 64, 4096), 64 * 1024 + 4096):
        ctx = B.ba_create(cfg, 0, room)
        tb = torch.empty(B.ba_segments_bytes(w.batch, w.n_blocks, w.n_tokens), dtype=torch.uint8, device="cuda")
        seg = B.ba_segment(ctx, np.asarray(w.block_lens, dtype=np.int32), np.asarray(w.seq_nblocks, dtype=np.int32), w.batch, w.n_blocks,
                           w.n_tokens, B.BA_MODE_BLOCK, tb)
        out, keys = torch.empty(Tf, w.n_q_heads, w.head_dim, device="cuda"), torch.empty(Tc, w.n_kv_heads, w.head_dim, dtype=torch.bfloat16, device="cuda")
        for k_out in (None, keys):
            B.ba_final_attend_fused(ctx, q, k, v, Tf, k_src, v_src, len(k_src), off, Tc, out, None, seg, B.BA_MODE_BLOCK, B.BA_OUT_F32, k_out=k_out)
            assert B.ba_last_device_status(ctx) == B.BA_OK
            check_attention(out.cpu().numpy(), o_ref)
        ref = torch.empty_like(keys)
        B.ba_reencode_k(ctx, k_src, off, len(k_src), ref, seg.cache_cu, seg.cache_delta, seg.n_cached_blocks, Tc)
        assert torch.equal(keys, ref)
        B.ba_destroy(ctx)


def _fused_kernel_cases():
    big = [_requests("stream_pool", 60, 95, (5, 20, 290), (33, 129), pool=True), _requests("stream_chunks", 60, 94, (4, 90, 300), (40, 140), heads=(8, 1, 64)),
           _requests("cluster", 1, 115, (9, 200, 340), (64, 64), heads=(32, 8, 128)), _requests("cluster_ragged", 5, 114, (3, 1, 500), (1, 70), heads=(8, 1, 64))]
    return big + [W.config1(), W.config2(), W.random_ragged(31, 3, 5, 200, 4, 2, 64), W.random_ragged(33, 3, 5, 200, 16, 2, 128),
                  _requests("odd_group", 2, 116, (6, 100, 300), (100, 140), heads=(6, 2, 64)), W.config5(4, 64, 6, 32)]


# The fused kernel itself, on caches that the call would take in two steps: a workspace without room for the keys leaves it
# no choice
@pytest.mark.parametrize("w", _fused_kernel_cases(), ids=lambda w: w.name)
@pytest.mark.parametrize("layout", [B.BA_ROPE_ADJACENT, B.BA_ROPE_HALF], ids=["adjacent", "half"])
def test_fused_kernel(w, layout):
    x, t = W.warm_inputs(w), ob.segment_tables(w.block_lens, w.seq_nblocks)
    k_src, v_src = (x[n] for n in (("k_pool", "v_pool") if w.pool_lens else ("k_cache", "v_cache")))
    off = x["src_off"] if w.pool_lens else None
    Tc, Tf = t["n_cached_tokens"], t["n_final_tokens"]
    lens = np.diff(t["cache_cu"])
    rows = np.concatenate([np.arange(o, o + n) for o, n in zip(off if off is not None else t["cache_cu"], lens)])
    f64 = W.bf16_bits_to_f64
    k_ref = ob.reencode_blocks(f64(k_src), off, t["cache_cu"], t["cache_delta"], w.rope_theta, layout)
    o_ref, lse_ref = ob.final_attend(f64(x["q_f"]), f64(x["k_f"]), f64(x["v_f"]), k_ref, f64(v_src)[rows], w.block_lens, w.seq_nblocks, B.BA_MODE_BLOCK)
    cfg = B.ba_config(w.n_q_heads, w.n_kv_heads, w.head_dim, layout, w.rope_theta, 0.0, 0)
    ctx = B.ba_create(cfg, 0, 64 * 1024 + Tc * w.n_kv_heads * w.head_dim * 3)
    tb = torch.empty(B.ba_segments_bytes(w.batch, w.n_blocks, w.n_tokens), dtype=torch.uint8, device="cuda")
    seg = B.ba_segment(ctx, np.asarray(w.block_lens, dtype=np.int32), np.asarray(w.seq_nblocks, dtype=np.int32), w.batch, w.n_blocks, w.n_tokens,
                       B.BA_MODE_BLOCK, tb)
    n0 = B.ba_launch_count(ctx)
    q, k, v, ks, vs = (R.bits_to_device(b) for b in (x["q_f"], x["k_f"], x["v_f"], k_src, v_src))
    d_off = torch.from_numpy(off).cuda() if off is not None else None
    o = torch.empty(Tf, w.n_q_heads, w.head_dim, device="cuda")
    lse = torch.empty(Tf, w.n_q_heads, device="cuda")
    B.ba_final_attend_fused(ctx, q, k, v, Tf, ks, vs, len(ks), d_off, Tc, o, lse, seg, B.BA_MODE_BLOCK, B.BA_OUT_F32)
    assert B.ba_last_device_status(ctx) == B.BA_OK
    assert B.ba_launch_count(ctx) - n0 == (1 if B.ba_last_attend_shape(ctx)["partials"] == 1 else 2)     # no re-encoding pass
    check_attention(o.cpu().numpy(), o_ref, lse.cpu().numpy(), lse_ref)
    # the same pool in pages of 16 rows
    if w.pool_lens is None:
        (kp, page_cu, page_idx, n_pages), vp = W.scatter_into_pages(k_src, lens, 16, 7), W.scatter_into_pages(v_src, lens, 16, 7)[0]
        keep = [R.bits_to_device(kp), R.bits_to_device(vp), torch.from_numpy(page_cu).cuda(), torch.from_numpy(page_idx).cuda()]
        o.fill_(float("nan"))
        B.ba_final_attend_fused_paged(ctx, q, k, v, Tf, keep[0], keep[1], B.make_page_table(16, n_pages, keep[2], keep[3]), Tc, o, lse, seg,
                                      B.BA_MODE_BLOCK, B.BA_OUT_F32)
        assert B.ba_last_device_status(ctx) == B.BA_OK
        check_attention(o.cpu().numpy(), o_ref, lse.cpu().numpy(), lse_ref)
    B.ba_destroy(ctx)


# Magnitudes of the cached keys that make a row's maximum grow from tile to tile, fall, or differ between the tiles that the two softmax
# groups of a CTA take, by far more than the factor the reference maximum may lag behind.
RAMPS = {"rising": lambda i, n, top: 1 + (top - 1) * i / n, "falling": lambda i, n, top: 1 + (top - 1) * (n - i) / n,
         "every_second_tile": lambda i, n, top: np.where(i // 128 % 2, top, 1.0)}


def _ramped_keys(w, x, ramp, top):
    n = len(x["k_cache"])
    return W.f32_to_bf16_bits(W.bf16_bits_to_f32(x["k_cache"]) * RAMPS[ramp](np.arange(n), n, top).astype(np.float32)[:, None, None])


# Clusters of one query tile (shared by both groups) and of whole items.  The oracle attends the keys as the GPU re-encoded them: at
# logits of hundreds their rounding to bf16 would weigh more than the attention's own error.  Bounds: those of the prefill's test.
@pytest.mark.parametrize("w", [_requests("one_query_tile", 2, 151, (9, 200, 340), (20, 32)),
                               _requests("whole_items", 1, 152, (20, 280, 320), (128, 128), heads=(32, 8, 128))], ids=lambda w: w.name)
@pytest.mark.parametrize("ramp", RAMPS)
def test_cluster_running_maximum(w, ramp):
    x, t, f64 = W.warm_inputs(w), ob.segment_tables(w.block_lens, w.seq_nblocks), W.bf16_bits_to_f64
    c = R.Context.for_workload(w)
    seg, buf = c.segment(w.block_lens, w.seq_nblocks, B.BA_MODE_BLOCK)
    keys = R.bits_to_device(_ramped_keys(w, x, ramp, 60.0))
    q, k, v, vc = (R.bits_to_device(x[n]) for n in ("q_f", "k_f", "v_f", "v_cache"))
    Tc, Tf = t["n_cached_tokens"], t["n_final_tokens"]
    k_re = torch.empty_like(keys)
    B.ba_reencode_k(c.ctx, keys, None, Tc, k_re, seg.cache_cu, seg.cache_delta, seg.n_cached_blocks, Tc)
    o, lse = torch.empty(Tf, w.n_q_heads, w.head_dim, device="cuda"), torch.empty(Tf, w.n_q_heads, device="cuda")
    B.ba_final_attend(c.ctx, q, k, v, Tf, k_re, vc, Tc, None, 0, o, lse, seg, B.BA_MODE_BLOCK, B.BA_OUT_F32)
    assert c.device_status() == B.BA_OK
    assert c.last_attend_shape()["partials"] == 1 and c.last_attend_shape()["balanced_tails"] == 0
    o_ref, lse_ref = ob.final_attend(f64(x["q_f"]), f64(x["k_f"]), f64(x["v_f"]), f64(R.device_to_bits(k_re)), f64(x["v_cache"]),
                                     w.block_lens, w.seq_nblocks, B.BA_MODE_BLOCK)
    d = np.abs(o.cpu().numpy() - o_ref)
    assert d.max() <= 2e-2 and d.mean() <= 1e-3 and np.linalg.norm(d) / np.linalg.norm(o_ref) <= 5e-3
    assert (np.abs(lse.cpu().numpy() - lse_ref) <= 2e-3 + 1e-5 * np.abs(lse_ref)).all()
    c.close()


# The fused kernel, on its own and in clusters, one and two query tiles.  It rounds the queries to bf16 once more after each block's
# rotation: a logit of standard deviation s is off by about s 2^-9 / sqrt(3) rms, 0.005 at s = 4, and a weight by as much of itself;
# five of those for the largest of 1e4 logits times values of up to 4 bound an element, twice the rms the whole.
@pytest.mark.parametrize("w", [_requests("short", 1, 153, (24, 250, 330), (9, 9), heads=(32, 8, 128)),
                               _requests("two_tiles", 1, 154, (24, 250, 330), (64, 64), heads=(32, 8, 128)),
                               _requests("cluster", 1, 155, (9, 200, 340), (30, 30), heads=(8, 2, 128))], ids=lambda w: w.name)
@pytest.mark.parametrize("ramp", RAMPS)
def test_fused_kernel_running_maximum(w, ramp):
    x, t, f64 = W.warm_inputs(w), ob.segment_tables(w.block_lens, w.seq_nblocks), W.bf16_bits_to_f64
    Tc, Tf = t["n_cached_tokens"], t["n_final_tokens"]
    bits = _ramped_keys(w, x, ramp, 4.0)
    k_ref = ob.reencode_blocks(f64(bits), None, t["cache_cu"], t["cache_delta"], w.rope_theta)
    o_ref, lse_ref = ob.final_attend(f64(x["q_f"]), f64(x["k_f"]), f64(x["v_f"]), k_ref, f64(x["v_cache"]), w.block_lens, w.seq_nblocks,
                                     B.BA_MODE_BLOCK)
    cfg = B.ba_config(w.n_q_heads, w.n_kv_heads, w.head_dim, 0, w.rope_theta, 0.0, 0)
    # (partial results have room, re-encoded keys have not)
    ctx = B.ba_create(cfg, 0, 64 * 1024 + Tc * w.n_kv_heads * w.head_dim * 3)
    tb = torch.empty(B.ba_segments_bytes(w.batch, w.n_blocks, w.n_tokens), dtype=torch.uint8, device="cuda")
    seg = B.ba_segment(ctx, np.asarray(w.block_lens, dtype=np.int32), np.asarray(w.seq_nblocks, dtype=np.int32), w.batch, w.n_blocks, w.n_tokens,
                       B.BA_MODE_BLOCK, tb)
    n0 = B.ba_launch_count(ctx)
    q, k, v, ks, vs = (R.bits_to_device(b) for b in (x["q_f"], x["k_f"], x["v_f"], bits, x["v_cache"]))
    o, lse = torch.empty(Tf, w.n_q_heads, w.head_dim, device="cuda"), torch.empty(Tf, w.n_q_heads, device="cuda")
    B.ba_final_attend_fused(ctx, q, k, v, Tf, ks, vs, Tc, None, Tc, o, lse, seg, B.BA_MODE_BLOCK, B.BA_OUT_F32)
    assert B.ba_last_device_status(ctx) == B.BA_OK
    assert B.ba_launch_count(ctx) - n0 == (1 if B.ba_last_attend_shape(ctx)["partials"] == 1 else 2)     # no re-encoding pass
    d = np.abs(o.cpu().numpy() - o_ref)
    assert d.max() <= 1e-1 and np.linalg.norm(d) / np.linalg.norm(o_ref) <= 1e-2
    assert np.abs(lse.cpu().numpy() - lse_ref).max() <= 2.5e-2
    B.ba_destroy(ctx)


# Tensors of one call whose cached tensor maps fall on the same slot of the context's 512: with the keys at 4096 places the
# map of the queries or of the values is met about 16 times.
def test_tensor_maps_that_share_a_slot():
    c = R.Context(4, 4, 64, 1e4)
    rows, places = 24, 4096
    gen = torch.Generator(device="cuda").manual_seed(7)
    q, k, v = (torch.randn(rows, 4, 64, generator=gen, device="cuda").bfloat16() for _ in range(3))
    seg, buf = c.segment(np.asarray([rows], dtype=np.int32), np.asarray([1], dtype=np.int32), B.BA_MODE_BLOCK, rows)
    room = torch.zeros(places * 128 + rows * 4 * 64, dtype=torch.bfloat16, device="cuda")
    want, o = torch.empty(rows, 4, 64, device="cuda"), torch.empty(rows, 4, 64, device="cuda")
    B.ba_block_prefill(c.ctx, q, k.float().bfloat16(), v, want, None, seg, B.BA_MODE_BLOCK, B.BA_OUT_F32)
    s = torch.einsum("ihd,jhd->hij", q.float(), k.float()) / 8.0
    p = s.masked_fill(torch.ones(rows, rows, device="cuda").triu(1).bool(), float("-inf")).softmax(-1)
    assert (want - torch.einsum("hij,jhd->ihd", p, v.float())).abs().max() < 1e-2
    wrong = torch.zeros((), dtype=torch.int64, device="cuda")
    for i in range(places):
        at = room[i * 128:i * 128 + rows * 4 * 64].view(rows, 4, 64)
        at.copy_(k)
        B.ba_block_prefill(c.ctx, q, at, v, o, None, seg, B.BA_MODE_BLOCK, B.BA_OUT_F32)
        wrong += (o != want).any()
    assert int(wrong) == 0
    assert c.device_status() == B.BA_OK
    c.close()
