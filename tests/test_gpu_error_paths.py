"""What the calls do with indexes that point outside their source, tables that do not hold and shapes at the edge of what a
step takes: reported, bounded and reproducible, as include/ba.h states.  Tolerances are those of the parity tests."""
import numpy as np
import pytest
import torch

from oracle import block_attention as ob
from paper_2409_15355_b200 import binding as B
from paper_2409_15355_b200 import runtime as R
from paper_2409_15355_b200 import workloads as W
from tests.test_gpu_parity import check_attention, check_reencoded, dev

pytestmark = pytest.mark.gpu


# ------------------------------------------------------------------ cached rows that point outside their source
def _fused(c, seg, x, ks, vs, source, Tc, Tf, w, k_out):
    """One fused call over rows at offsets (`source` an int32 tensor) or pages (a page table)."""
    o = torch.full((Tf, w.n_q_heads, w.head_dim), float("nan"), device="cuda")
    lse = torch.full((Tf, w.n_q_heads), float("nan"), device="cuda")
    q, k, v = (dev(x[n]) for n in ("q_f", "k_f", "v_f"))
    if isinstance(source, B.ba_page_table):
        B.ba_final_attend_fused_paged(c.ctx, q, k, v, Tf, ks, vs, source, Tc, o, lse, seg, B.BA_MODE_BLOCK, B.BA_OUT_F32, k_out=k_out)
    else:
        B.ba_final_attend_fused(c.ctx, q, k, v, Tf, ks, vs, len(ks), source, Tc, o, lse, seg, B.BA_MODE_BLOCK, B.BA_OUT_F32, k_out=k_out)
    return o, lse


@pytest.mark.parametrize("layout", [B.BA_ROPE_ADJACENT, B.BA_ROPE_HALF], ids=["adjacent", "half"])
@pytest.mark.parametrize("paged", [False, True], ids=["offsets", "pages"])
@pytest.mark.parametrize("with_k_out", [False, True], ids=["workspace", "k_out"])
def test_fused_call_reads_zeros_for_rows_outside_the_source(layout, paged, with_k_out):
    """Rows whose offset or page lies outside the source count as zeros in the fused call, whichever way it takes: nothing
    of an earlier call (here NaN keys and values) shows in the result, and it is the same from run to run."""
    w = W.Workload("outside", 8, 2, 128, 1e4, [64, 33, 100, 64, 40], [5], seed=141)
    lens, t, x = w.block_lens[:4], ob.segment_tables(w.block_lens, w.seq_nblocks), W.warm_inputs(w)
    Tc, Tf, f64 = t["n_cached_tokens"], t["n_final_tokens"], W.bf16_bits_to_f64
    c = R.Context(8, 2, 128, 1e4, rope_layout=layout)
    seg, buf = c.segment(w.block_lens, w.seq_nblocks, B.BA_MODE_BLOCK)
    if paged:
        (kp, page_cu, page_idx, n_pages), vp = W.scatter_into_pages(x["k_cache"], lens, 16, 3), W.scatter_into_pages(x["v_cache"], lens, 16, 3)[0]
        bad_idx = page_idx.copy()
        bad_idx[2], bad_idx[5], bad_idx[-1] = 10 ** 6, -2, n_pages
        keep = [torch.from_numpy(a).cuda() for a in (page_cu, page_idx, bad_idx)]
        good, bad = (B.make_page_table(16, n_pages, keep[0], i) for i in keep[1:])
        rows = np.concatenate([bad_idx[page_cu[i] + np.arange(n) // 16] * 16 + np.arange(n) % 16 for i, n in enumerate(lens)])
    else:
        kp, vp = x["k_cache"], x["v_cache"]
        off = np.asarray([0, -5, Tc - 30, 1 << 30], dtype=np.int32)        # in place, partly in front, partly behind, far outside
        keep = [torch.from_numpy(a).cuda() for a in (t["cache_cu"][:-1].astype(np.int32), off)]
        good, bad = keep
        rows = np.concatenate([o.astype(np.int64) + np.arange(n) for o, n in zip(off, lens)])
    inside = (rows >= 0) & (rows < len(kp))
    assert inside.any() and not inside.all()
    k64, v64 = (np.where(inside[:, None, None], f64(p)[np.where(inside, rows, 0)], 0.0) for p in (kp, vp))
    k_ref = ob.reencode_blocks(k64, None, t["cache_cu"], t["cache_delta"], 1e4, layout)
    o_ref, lse_ref = ob.final_attend(f64(x["q_f"]), f64(x["k_f"]), f64(x["v_f"]), k_ref, v64, w.block_lens, w.seq_nblocks)
    k, v = dev(kp), dev(vp)
    nan = torch.full_like(k, float("nan"))
    k_out = torch.empty(Tc, 2, 128, dtype=torch.bfloat16, device="cuda") if with_k_out else None
    got = []
    for _ in range(2):
        if with_k_out:
            k_out.fill_(float("nan"))
        _fused(c, seg, x, nan, nan, good, Tc, Tf, w, k_out)                # an earlier call with other contents
        got.append(_fused(c, seg, x, k, v, bad, Tc, Tf, w, k_out))
        # written keys are ba_reencode_k's, which reports such rows; a call that only attends reads zeros and says nothing
        assert c.device_status() == (B.BA_ERR_INVALID_ARG if with_k_out else B.BA_OK)
        check_attention(got[-1][0].cpu().numpy(), o_ref, got[-1][1].cpu().numpy(), lse_ref)
    assert torch.equal(got[0][0], got[1][0]) and torch.equal(got[0][1], got[1][1])
    if with_k_out:
        check_reencoded(R.device_to_bits(k_out), k_ref)
        assert not k_out[torch.from_numpy(~inside).cuda()].any()
    c.close()


# ------------------------------------------------------------------ more KV heads than a re-encoding row has threads for
@pytest.mark.parametrize("heads,layout,wide", [((40, 40, 128), B.BA_ROPE_ADJACENT, True), ((32, 32, 128), B.BA_ROPE_ADJACENT, False),
                                               ((40, 40, 128), B.BA_ROPE_HALF, False), ((65, 65, 128), B.BA_ROPE_HALF, True),
                                               ((66, 66, 64), B.BA_ROPE_ADJACENT, True)], ids=str)
def test_fused_call_takes_rows_wider_than_the_reencoding_kernel(heads, layout, wide):
    """n_kv_heads * head_dim above what ba_reencode_k takes (it says so): the fused call without k_out still works, as the
    rotation is then applied to the queries; with k_out it is refused like ba_reencode_k."""
    w = W.Workload("wide", *heads, 1e4, [70, 33, 20], [3], seed=151)
    t, x, f64 = ob.segment_tables(w.block_lens, w.seq_nblocks), W.warm_inputs(w), W.bf16_bits_to_f64
    Tc, Tf = t["n_cached_tokens"], t["n_final_tokens"]
    c = R.Context(*heads, 1e4, rope_layout=layout, max_q_rows=4096)
    seg, buf = c.segment(w.block_lens, w.seq_nblocks, B.BA_MODE_BLOCK)
    k, v = dev(x["k_cache"]), dev(x["v_cache"])
    k_ref = ob.reencode_blocks(f64(x["k_cache"]), None, t["cache_cu"], t["cache_delta"], 1e4, layout)
    o_ref, lse_ref = ob.final_attend(f64(x["q_f"]), f64(x["k_f"]), f64(x["v_f"]), k_ref, f64(x["v_cache"]), w.block_lens, w.seq_nblocks)
    (kp, page_cu, page_idx, n_pages), vp = W.scatter_into_pages(x["k_cache"], w.block_lens[:2], 16, 3), W.scatter_into_pages(x["v_cache"], w.block_lens[:2], 16, 3)[0]
    d_cu, d_idx = torch.from_numpy(page_cu).cuda(), torch.from_numpy(page_idx).cuda()
    for ks, vs, source in ((k, v, None), (dev(kp), dev(vp), B.make_page_table(16, n_pages, d_cu, d_idx))):
        o, lse = _fused(c, seg, x, ks, vs, source, Tc, Tf, w, None)
        assert c.device_status() == B.BA_OK
        check_attention(o.cpu().numpy(), o_ref, lse.cpu().numpy(), lse_ref)
        k_out = torch.empty_like(k)
        if wide:
            with pytest.raises(B.BaError) as e:
                _fused(c, seg, x, ks, vs, source, Tc, Tf, w, k_out)
            assert e.value.status == B.BA_ERR_UNSUPPORTED
        else:
            _fused(c, seg, x, ks, vs, source, Tc, Tf, w, k_out)
            check_reencoded(R.device_to_bits(k_out), k_ref)
    c.close()


# ------------------------------------------------------------------ tables of lengths that do not add up, page lists too short
@pytest.mark.parametrize("fault", ["tokens", "zero_length", "block_counts"])
def test_split_keys_over_inconsistent_tables_leave_the_output_alone(fault):
    """Lengths on the device that do not add up leave the item tables as they were (here: those of an earlier call).  The keys of a
    short final block are split over several CTAs, whose results a second kernel merges: neither touches the output."""
    w = W.Workload("tables", 8, 2, 64, 1e4, [64, 33, 300, 40], [4], seed=161)
    x = W.warm_inputs(w)
    Tf, Tc = 40, w.n_tokens - 40
    c = R.Context(8, 2, 64, 1e4)
    q, k, v, kc, vc = (dev(x[n]) for n in ("q_f", "k_f", "v_f", "k_cache", "v_cache"))
    o = torch.full((Tf, 8, 64), 7.0, device="cuda")
    lse = torch.full((Tf, 8), 7.0, device="cuda")
    lens, nb = torch.tensor(w.block_lens, dtype=torch.int32, device="cuda"), torch.tensor([4], dtype=torch.int32, device="cuda")
    buf = torch.zeros(B.ba_segments_bytes(1, 4, w.n_tokens), dtype=torch.uint8, device="cuda")
    seg = B.ba_segment(c.ctx, lens, nb, 1, 4, w.n_tokens, B.BA_MODE_BLOCK, buf)
    B.ba_final_attend(c.ctx, q, k, v, Tf, kc, vc, Tc, None, 0, o, lse, seg, B.BA_MODE_BLOCK, B.BA_OUT_F32)
    assert c.device_status() == B.BA_OK and c.last_attend_shape()["partials"] > 1
    assert torch.isfinite(o).all() and not (o == 7.0).any()
    o.fill_(7.0); lse.fill_(7.0)
    if fault == "tokens":
        lens[1] += 1
    elif fault == "zero_length":
        lens[1] = 0
    else:
        nb[0] = 3
    seg = B.ba_segment(c.ctx, lens, nb, 1, 4, w.n_tokens, B.BA_MODE_BLOCK, buf)
    assert c.device_status() == B.BA_ERR_INVALID_ARG
    B.ba_final_attend(c.ctx, q, k, v, Tf, kc, vc, Tc, None, 0, o, lse, seg, B.BA_MODE_BLOCK, B.BA_OUT_F32)
    torch.cuda.synchronize()
    assert c.last_attend_shape()["partials"] > 1
    assert (o == 7.0).all() and (lse == 7.0).all()
    c.close()


def _paged_request():
    w = W.Workload("tables", 8, 2, 64, 1e4, [64, 33, 100, 40], [4], seed=161)
    t, x = ob.segment_tables(w.block_lens, w.seq_nblocks), W.warm_inputs(w)
    (kp, page_cu, page_idx, n_pages), vp = W.scatter_into_pages(x["k_cache"], w.block_lens[:3], 16, 3), W.scatter_into_pages(x["v_cache"], w.block_lens[:3], 16, 3)[0]
    d_cu, d_idx = torch.from_numpy(page_cu).cuda(), torch.from_numpy(page_idx).cuda()
    return w, t, x, dev(kp), dev(vp), d_cu, d_idx, n_pages


@pytest.mark.parametrize("fault", ["tokens", "zero_length", "block_counts"])
def test_calls_over_inconsistent_tables_report_and_move_nothing(fault):
    """Lengths on the device that do not add up: ba_segment leaves the tables unwritten (here: a buffer of a large pattern).
    Every call that walks them reports it and touches none of its outputs, the re-encoding step of a fused call among them."""
    w, t, x, kp, vp, d_cu, d_idx, n_pages = _paged_request()
    Tc, Tf = t["n_cached_tokens"], t["n_final_tokens"]
    c = R.Context(8, 2, 64, 1e4)
    lens, nb, T = torch.tensor(w.block_lens, dtype=torch.int32, device="cuda"), torch.tensor([4], dtype=torch.int32, device="cuda"), w.n_tokens
    buf = torch.full((B.ba_segments_bytes(1, 4, T),), 0x3f, dtype=torch.uint8, device="cuda")
    if fault == "tokens":
        lens[1] += 1
    elif fault == "zero_length":
        lens[1] = 0
    else:
        nb[0] = 3
    seg = B.ba_segment(c.ctx, lens, nb, 1, 4, T, B.BA_MODE_BLOCK, buf)
    assert c.device_status() == B.BA_ERR_INVALID_ARG
    pages = B.make_page_table(16, n_pages, d_cu, d_idx)
    q, k, v = (dev(x[n]) for n in ("q_f", "k_f", "v_f"))
    k_src, v_src = dev(x["k_cache"]), dev(x["v_cache"])
    o = torch.full((Tf, 8, 64), 7.0, device="cuda")
    for with_k_out in (False, True):
        for call in ("fused", "paged", "reencode_paged", "reencode", "deferred"):
            if call in ("reencode_paged", "reencode", "deferred") and not with_k_out:
                continue
            keys = torch.full((Tc, 2, 64), 7.0, dtype=torch.bfloat16, device="cuda")
            k_out = keys if with_k_out else None
            if call == "fused":
                B.ba_final_attend_fused(c.ctx, q, k, v, Tf, k_src, v_src, Tc, None, Tc, o, None, seg, B.BA_MODE_BLOCK, B.BA_OUT_F32, k_out=k_out)
            elif call == "paged":
                B.ba_final_attend_fused_paged(c.ctx, q, k, v, Tf, kp, vp, pages, Tc, o, None, seg, B.BA_MODE_BLOCK, B.BA_OUT_F32, k_out=k_out)
            elif call == "reencode_paged":
                B.ba_reencode_k_paged(c.ctx, kp, pages, keys, seg.cache_cu, seg.cache_delta, 3, Tc)
            elif call == "reencode":
                B.ba_reencode_k(c.ctx, k_src, None, Tc, keys, seg.cache_cu, seg.cache_delta, 3, Tc)
            else:
                B.ba_reencode_k_deferred(c.ctx, k_src, None, Tc, keys, seg.cache_cu, seg.cache_delta, 3, Tc)
                B.ba_final_attend(c.ctx, q, k, v, Tf, k_src, v_src, Tc, None, 0, o, None, seg, B.BA_MODE_BLOCK, B.BA_OUT_F32)
            assert c.device_status() == B.BA_ERR_INVALID_ARG, call
            assert (o == 7.0).all() and (keys == 7.0).all(), call
    c.close()


def test_page_list_shorter_than_its_block():
    """Rows past the end of their block's page list are rows outside the source; the next list's entries are not theirs."""
    w, t, x, kp, vp, d_cu, d_idx, n_pages = _paged_request()
    Tc = t["n_cached_tokens"]
    c = R.Context(8, 2, 64, 1e4)
    seg, buf = c.segment(w.block_lens, w.seq_nblocks, B.BA_MODE_BLOCK)
    want, got = (torch.zeros(Tc, 2, 64, dtype=torch.bfloat16, device="cuda") for _ in range(2))
    B.ba_reencode_k_paged(c.ctx, kp, B.make_page_table(16, n_pages, d_cu, d_idx), want, seg.cache_cu, seg.cache_delta, 3, Tc)
    assert c.device_status() == B.BA_OK
    short = d_cu.clone()
    short[-1] -= 2                                                         # the last block: rows 80 .. 99 have no page
    for call in range(2):
        got.zero_()
        own = torch.from_numpy(t["cache_delta"].astype(np.int32)).cuda()   # (the tables' own array, then a caller's)
        B.ba_reencode_k_paged(c.ctx, kp, B.make_page_table(16, n_pages, short, d_idx), got, seg.cache_cu, own if call else seg.cache_delta, 3, Tc)
        assert c.device_status() == B.BA_ERR_INVALID_ARG
        assert torch.equal(got[:Tc - 20], want[:Tc - 20]) and not got[Tc - 20:].any()
    c.close()


def test_prefill_over_tables_rebuilt_with_longer_final_blocks():
    """A prefill keeps partial results of the final blocks' rows, in room for as many as its ba_segments says.  When the buffer has
    been rebuilt since with more of them, the call reports it and writes nothing."""
    a, b = [300] * 9 + [65], [100] * 9 + [1865]
    w = W.Workload("rebuilt", 32, 8, 128, 1e4, a, [10], seed=171)
    x = [dev(v) for v in W.prefill_inputs(w)]
    c = R.Context.for_workload(w)
    seg, buf = c.segment(a, [10], B.BA_MODE_BLOCK)
    o = torch.full((w.n_tokens, 32, 128), 7.0, device="cuda")
    B.ba_block_prefill(c.ctx, *x, o, None, seg, B.BA_MODE_BLOCK, B.BA_OUT_F32)
    assert c.device_status() == B.BA_OK and c.last_attend_shape()["partials"] > 1
    o.fill_(7.0)
    B.ba_segment(c.ctx, np.asarray(b, dtype=np.int32), np.asarray([10], dtype=np.int32), 1, 10, w.n_tokens, B.BA_MODE_BLOCK, buf)
    B.ba_block_prefill(c.ctx, *x, o, None, seg, B.BA_MODE_BLOCK, B.BA_OUT_F32)
    assert c.device_status() == B.BA_ERR_SHAPE
    assert (o == 7.0).all()
    c.close()
