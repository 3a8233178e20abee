"""The work a user of this library has it do, as measurable cases.

Every case is one pass of a serving or training program through the public entry points (runtime.Context and
the functions of binding): the tables of a batch of prompts, then the attention calls of some layers.  A program
keeps its context, its caches and its output buffers; the block lengths of a prompt arrive on the host with
the request, so ba_segment belongs to the pass.  Values are i.i.d. N(0, 1) in bf16, like the seeded inputs of
workloads.py; the lengths of a case follow from its `lens_seed`.

Paths
  warm     re-encode the cached keys of every layer, then the final block attends (two calls a layer);
           two_streams: layer l + 1 is re-encoded on a second stream while layer l attends, as bench.py does
  fused    the same in one call a layer; k_out: the re-encoded keys are written back for the decode steps
  pool     as warm, with cached blocks gathered from a shared pool by offset and values read there in place
  paged    as fused, with keys and values in fixed-size pages of a shared pool
  edit     edited blocks are encoded again: a packed buffer of one-block prompts
  cold     a prompt is encoded for the first time and its keys are rotated back to position zero for the cache
  prefill  a packed batch of prompts, attention forward
  train    the same with log-sum-exp, and its backward pass
"""
import math
import random

import numpy as np
import torch

from paper_2409_15355_b200 import binding as B
from paper_2409_15355_b200 import runtime as R

DEVICE = "cuda:0"


def _case(name, path, shape, blocks, lo, hi, final, lens_seed, batch=1, layers=1, seq_len=0, mode="block", rope="adjacent",
          out="bf16", **more):
    """blocks: cached blocks a sequence, lengths U[lo, hi], then a final block of `final` tokens.  seq_len > 0:
    lengths U[lo, hi] until the sequence has seq_len tokens instead, its last block being the final one."""
    c = {"path": path, "q_heads": shape[0], "kv_heads": shape[1], "head_dim": shape[2], "batch": batch,
         "blocks": blocks, "lo": lo, "hi": hi, "final": final, "seq_len": seq_len, "layers": layers, "mode": mode, "rope": rope,
         "out": out, "lens_seed": lens_seed, "two_streams": False, "k_out": False, "pool_blocks": 0, "page_rows": 0}
    c.update(more)
    if name:
        c["name"] = name
    return c


LLAMA = (32, 8, 128)   # attention shape of Llama-3-8B


def listed():
    return [
        # the smallest request: four passages of 64 tokens and a question, one layer of a small model; all latency
        _case("tiny_request", "warm", (4, 2, 64), 4, 64, 64, 32, 1001, out="f32"),
        # an ordinary retrieval prompt: ten passages of 128-384 tokens and a question, every layer of the model
        _case("rag_request", "warm", LLAMA, 10, 128, 384, 64, 2002, layers=32),
        # the long prompt of the benchmark: 32 passages of 1000 tokens, a final block of 768, all layers, two streams
        _case("long_request", "warm", LLAMA, 32, 1000, 1000, 768, 3003, layers=32, two_streams=True),
        # the same cache under a short question, in one call a layer; keys written back for decoding
        _case("long_short_query", "fused", LLAMA, 32, 1000, 1000, 64, 3004, layers=8, k_out=True),
        # sixteen requests served together from a pool of 512 passages
        _case("pool_serving", "pool", LLAMA, 20, 50, 500, 128, 5005, batch=16, layers=4, pool_blocks=512),
        # eight requests served from a paged pool by the fused call, rotary halves, ragged everything
        _case("paged_serving", "paged", LLAMA, 12, 37, 611, 101, 6006, batch=8, layers=4, pool_blocks=160, page_rows=64,
              rope="half"),
        # seven passages of a cached prompt were edited: they are encoded again, layer by layer
        _case("edited_blocks", "edit", LLAMA, 7, 50, 500, 0, 7007, layers=8),
        # a retrieval prompt seen for the first time, encoded block by block and put into the cache
        _case("cold_request", "cold", LLAMA, 18, 100, 700, 96, 8008, layers=8),
        # a batch of long prompts encoded in one launch
        _case("cold_batch", "prefill", LLAMA, 0, 64, 2048, 0, 4004, batch=8, seq_len=16384),
        # the long prompt under ordinary causal attention (the fine-tuned model runs under either mask)
        _case("cold_full_causal", "prefill", LLAMA, 32, 1000, 1000, 768, 3005, mode="full"),
        # block fine-tuning: forward and backward of a batch of long prompts
        _case("finetune_batch", "train", LLAMA, 0, 64, 2048, 0, 4004, batch=8, seq_len=16384),
        # the same for a small model with an odd group of heads, short ragged prompts, gradients in fp32
        _case("finetune_small", "train", (6, 2, 64), 5, 30, 300, 75, 9009, batch=3, out="f32"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    path = rng.choice(["warm", "warm", "fused", "fused", "pool", "paged", "edit", "cold", "prefill", "prefill", "train", "train"])
    small = rng.random() < 0.25
    shape = rng.choice([(4, 2, 64), (6, 2, 64), (8, 2, 128), (8, 1, 128), (4, 4, 128)]) if small else LLAMA
    seed = rng.randrange(1, 1 << 20)
    rope = rng.choice(["adjacent", "adjacent", "half"])
    mode = rng.choice(["block", "block", "full"])
    out = rng.choice(["bf16", "bf16", "bf16", "f32"])
    lo = rng.randrange(1, 200)
    hi = _log_int(rng, max(lo, 64), 2048)
    if path in ("warm", "fused"):
        blocks = _log_int(rng, 2, 40)
        return _case(None, path, shape, blocks, lo, hi, _log_int(rng, 1, 1024), seed, layers=rng.choice([1, 2, 4, 8]), rope=rope,
                     out=out, mode=mode, two_streams=path == "warm" and rng.random() < 0.3,
                     k_out=path == "fused" and rng.random() < 0.6)
    if path in ("pool", "paged"):
        hi = min(hi, 800)
        lo = min(lo, hi)
        return _case(None, path, shape, rng.randrange(3, 24), lo, hi, _log_int(rng, 1, 256), seed, batch=_log_int(rng, 1, 24),
                     layers=rng.choice([1, 2, 4]), rope=rope, out=out, mode=mode, pool_blocks=rng.randrange(24, 300),
                     page_rows=rng.choice([16, 32, 64, 128, 256]) if path == "paged" else 0,
                     k_out=path == "paged" and rng.random() < 0.5)
    if path == "edit":
        return _case(None, path, shape, _log_int(rng, 1, 24), lo, min(hi, 900) if hi > lo else lo, 0, seed, layers=rng.choice([1, 4, 8]),
                     out=out)
    if path == "cold":
        return _case(None, path, shape, _log_int(rng, 2, 40), lo, hi, _log_int(rng, 1, 512), seed, layers=rng.choice([1, 4, 8]), rope=rope,
                     out=out, mode=mode)
    batch = _log_int(rng, 1, 8)
    return _case(None, path, shape, 0, lo, hi, 0, seed, batch=batch, seq_len=_log_int(rng, 200, 16384), out=out,
                 mode=mode if batch <= 2 else "block")


# ------------------------------------------------------------------------------------------------ the prompts of a case
class _Prompts:
    """Block lengths of the batch in prompt order, blocks a sequence, and (pool paths) the pool's blocks."""

    def __init__(self, c):
        rng = random.Random(c["lens_seed"])
        self.pool_lens = [rng.randint(c["lo"], c["hi"]) for _ in range(c["pool_blocks"])]
        self.pool_idx, seqs = [], []
        for _ in range(c["batch"]):
            if c["path"] == "edit":
                seqs += [[rng.randint(c["lo"], c["hi"])] for _ in range(c["blocks"])]
            elif c["seq_len"]:
                s = []
                while sum(s) < c["seq_len"]:
                    s.append(min(rng.randint(c["lo"], c["hi"]), c["seq_len"] - sum(s)))
                seqs.append(s)
            elif c["pool_blocks"]:
                pick = [rng.randrange(c["pool_blocks"]) for _ in range(c["blocks"])]
                self.pool_idx += pick
                seqs.append([self.pool_lens[i] for i in pick] + [c["final"]])
            else:
                seqs.append([rng.randint(c["lo"], c["hi"]) for _ in range(c["blocks"])] + [c["final"]])
        self.seqs = seqs
        self.lens = np.asarray([n for s in seqs for n in s], dtype=np.int32)
        self.n_blocks = np.asarray([len(s) for s in seqs], dtype=np.int32)
        self.tokens = int(self.lens.sum())
        self.final_rows = sum(s[-1] for s in seqs)
        self.cache_rows = self.tokens - self.final_rows

    def pairs(self, final_only, full):
        """(query, key) pairs the mask allows, per head."""
        n = 0
        for s in self.seqs:
            total, fin = sum(s), s[-1]
            if final_only:
                n += fin * (total - fin) + fin * (fin + 1) // 2
            elif full:
                n += total * (total + 1) // 2
            else:
                n += sum(b * (b + 1) // 2 for b in s) + fin * (total - fin)
        return n


def _pages(c, p):
    """Page list of every cached block: the pool's blocks own pages in shuffled order."""
    rows = c["page_rows"]
    rng = random.Random(c["lens_seed"] + 1)
    need = [-(-n // rows) for n in p.pool_lens]
    order = list(range(sum(need)))
    rng.shuffle(order)
    own, at = [], 0
    for n in need:
        own.append(order[at:at + n])
        at += n
    lists = [own[i] for i in p.pool_idx]
    cu = np.concatenate([[0], np.cumsum([len(x) for x in lists])]).astype(np.int32)
    return cu, np.asarray([g for x in lists for g in x], dtype=np.int32), len(order)


# ------------------------------------------------------------------------------------------------ one pass
class _State:
    pass


def prepare(case, seed):
    c, s = case, _State()
    s.c, s.p = c, _Prompts(c)
    p = s.p
    hq, hkv, d, layers = c["q_heads"], c["kv_heads"], c["head_dim"], c["layers"]
    gen = torch.Generator(device=DEVICE)
    gen.manual_seed(seed)
    bf16 = torch.bfloat16
    s.out_type, s.out_dtype = (B.BA_OUT_F32, torch.float32) if c["out"] == "f32" else (B.BA_OUT_BF16, bf16)
    s.mode = B.BA_MODE_FULL if c["mode"] == "full" else B.BA_MODE_BLOCK
    s.ctx = R.Context(hq, hkv, d, 10000.0 if d == 64 else 500000.0, B.BA_ROPE_HALF if c["rope"] == "half" else B.BA_ROPE_ADJACENT)

    def values(*shape):
        return torch.randn(*shape, generator=gen, device=DEVICE, dtype=bf16)

    def room(*shape, dtype=bf16):
        return torch.empty(*shape, device=DEVICE, dtype=dtype)

    if c["path"] in ("warm", "fused", "pool", "paged"):
        s.q, s.k, s.v = values(layers, p.final_rows, hq, d), values(layers, p.final_rows, hkv, d), values(layers, p.final_rows, hkv, d)
        s.o = room(layers, p.final_rows, hq, d, dtype=s.out_dtype)
        rows = p.cache_rows
        if c["path"] == "pool":
            rows = sum(p.pool_lens)
            first = np.concatenate([[0], np.cumsum(p.pool_lens)])
            s.src_off = torch.from_numpy(np.asarray([first[i] for i in p.pool_idx], dtype=np.int32)).to(DEVICE)
        if c["path"] == "paged":
            cu, idx, n_pages = _pages(c, p)
            s.page_cu, s.page_idx = torch.from_numpy(cu).to(DEVICE), torch.from_numpy(idx).to(DEVICE)
            s.pages = B.make_page_table(c["page_rows"], n_pages, s.page_cu, s.page_idx)
            rows = n_pages * c["page_rows"]
        s.k_cache, s.v_cache = values(layers, rows, hkv, d), values(layers, rows, hkv, d)
        s.k_new = room(layers, p.cache_rows, hkv, d) if c["path"] in ("warm", "pool") or c["k_out"] else None
        if c["two_streams"]:
            s.side = torch.cuda.Stream(device=DEVICE, priority=0)
            s.main = torch.cuda.Stream(device=DEVICE, priority=-1)
    else:
        s.q, s.k, s.v = values(layers, p.tokens, hq, d), values(layers, p.tokens, hkv, d), values(layers, p.tokens, hkv, d)
        s.o = room(layers, p.tokens, hq, d, dtype=bf16 if c["path"] == "train" else s.out_dtype)
        if c["path"] == "cold":
            s.k_fill = room(layers, p.cache_rows, hkv, d)
            start = np.concatenate([[0], np.cumsum(p.lens[:-1])])[:-1]
            s.back = torch.from_numpy((-start).astype(np.int32)).to(DEVICE)
        if c["path"] == "train":
            s.grad = values(layers, p.tokens, hq, d)
            s.lse = room(layers, p.tokens, hq, dtype=torch.float32)
            s.dq = room(layers, p.tokens, hq, d, dtype=s.out_dtype)
            s.dk, s.dv = room(layers, p.tokens, hkv, d, dtype=s.out_dtype), room(layers, p.tokens, hkv, d, dtype=s.out_dtype)
    return s


def _warm(s, seg):
    p, ctx = s.p, s.ctx.ctx
    for l in range(s.c["layers"]):
        B.ba_reencode_k(ctx, s.k_cache[l], None, p.cache_rows, s.k_new[l], seg.cache_cu, seg.cache_delta, seg.n_cached_blocks,
                        p.cache_rows)
        B.ba_final_attend(ctx, s.q[l], s.k[l], s.v[l], p.final_rows, s.k_new[l], s.v_cache[l], p.cache_rows, None, 0, s.o[l], None, seg,
                          s.mode, s.out_type)


def _warm_two_streams(s):
    """Layer l + 1 is re-encoded on the side stream while layer l attends on the main one."""
    p, ctx, layers = s.p, s.ctx.ctx, s.c["layers"]
    s.main.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(s.main):
        s.tables = s.ctx.segment(p.lens, p.n_blocks, s.mode, p.tokens)
        seg = s.tables[0]
        s.side.wait_stream(s.main)
        attended = []

        def attend(l, keys_ready):
            s.main.wait_event(keys_ready)
            B.ba_final_attend(ctx, s.q[l], s.k[l], s.v[l], p.final_rows, s.k_new[l], s.v_cache[l], p.cache_rows, None, 0, s.o[l], None,
                              seg, s.mode, s.out_type)
            attended.append(s.main.record_event())

        ready = None
        for l in range(layers):
            if l >= 2:
                s.side.wait_event(attended[l - 2])
            B.ba_reencode_k(ctx, s.k_cache[l], None, p.cache_rows, s.k_new[l], seg.cache_cu, seg.cache_delta, seg.n_cached_blocks,
                            p.cache_rows, stream=s.side)
            now = s.side.record_event()
            if l:
                attend(l - 1, ready)
            ready = now
        attend(layers - 1, ready)
    torch.cuda.current_stream().wait_stream(s.main)


def run(s):
    c, p, ctx = s.c, s.p, s.ctx.ctx
    path, layers = c["path"], c["layers"]
    if c["two_streams"]:
        _warm_two_streams(s)
        return {"o": s.o, "k": s.k_new}
    s.tables = s.ctx.segment(p.lens, p.n_blocks, s.mode, p.tokens)
    seg = s.tables[0]
    if path == "warm":
        _warm(s, seg)
        return {"o": s.o, "k": s.k_new}
    if path == "fused":
        for l in range(layers):
            B.ba_final_attend_fused(ctx, s.q[l], s.k[l], s.v[l], p.final_rows, s.k_cache[l], s.v_cache[l], p.cache_rows, None,
                                    p.cache_rows, s.o[l], None, seg, s.mode, s.out_type, k_out=s.k_new[l] if c["k_out"] else None)
        return {"o": s.o, "k": s.k_new}
    if path == "pool":
        rows = s.k_cache.shape[1]
        for l in range(layers):
            B.ba_reencode_k(ctx, s.k_cache[l], s.src_off, rows, s.k_new[l], seg.cache_cu, seg.cache_delta, seg.n_cached_blocks,
                            p.cache_rows)
            B.ba_final_attend(ctx, s.q[l], s.k[l], s.v[l], p.final_rows, s.k_new[l], s.v_cache[l], p.cache_rows, s.src_off, rows,
                              s.o[l], None, seg, s.mode, s.out_type)
        return {"o": s.o, "k": s.k_new}
    if path == "paged":
        for l in range(layers):
            B.ba_final_attend_fused_paged(ctx, s.q[l], s.k[l], s.v[l], p.final_rows, s.k_cache[l], s.v_cache[l], s.pages, p.cache_rows,
                                          s.o[l], None, seg, s.mode, s.out_type, k_out=s.k_new[l] if c["k_out"] else None)
        return {"o": s.o, "k": s.k_new}
    for l in range(layers):
        lse = s.lse[l] if path == "train" else None
        B.ba_block_prefill(ctx, s.q[l], s.k[l], s.v[l], s.o[l], lse, seg, s.mode, B.BA_OUT_BF16 if path == "train" else s.out_type)
        if path == "cold":
            B.ba_reencode_k(ctx, s.k[l], None, p.tokens, s.k_fill[l], seg.cache_cu, s.back, seg.n_cached_blocks, p.cache_rows)
        if path == "train":
            B.ba_block_prefill_bwd(ctx, s.q[l], s.k[l], s.v[l], s.o[l], lse, s.grad[l], s.dq[l], s.dk[l], s.dv[l], seg, s.mode,
                                   s.out_type)
    if path == "cold":
        return {"o": s.o, "k": s.k_fill}
    if path == "train":
        return {"o": s.o, "lse": s.lse, "dq": s.dq, "dk": s.dk, "dv": s.dv}
    return {"o": s.o}


def work(case):
    c, p = case, _Prompts(case)
    hq, hkv, d = c["q_heads"], c["kv_heads"], c["head_dim"]
    path, wide = c["path"], 4 if c["out"] == "f32" else 2
    q_row, kv_row = hq * d, hkv * d
    final_only = path in ("warm", "fused", "pool", "paged")
    flops = 4.0 * d * hq * p.pairs(final_only, c["mode"] == "full")
    if final_only:
        fresh = p.cache_rows
        if c["pool_blocks"]:                                   # a passage that several requests use is read once
            fresh = sum(p.pool_lens[i] for i in set(p.pool_idx))
        n = p.final_rows * (2 * q_row + wide * q_row + 4 * kv_row) + fresh * 4 * kv_row
        if path in ("warm", "pool") or c["k_out"]:
            n += p.cache_rows * 2 * kv_row
    else:
        n = p.tokens * (2 * q_row + 4 * kv_row)
        if path == "train":                                    # o and lse are written, the gradients of o read, dq, dk, dv written
            n += p.tokens * (2 * q_row + 4 * hq + 2 * q_row + wide * (q_row + 2 * kv_row))
            flops *= 3.5
        else:
            n += p.tokens * wide * q_row
        if path == "cold":
            n += p.cache_rows * 2 * kv_row
    return {"bytes": float(n * c["layers"]), "flops": flops * c["layers"]}


def tolerance(case):
    """Against the same path in fp64 (bf16 operands, P, dS and stores; fp32 sums) the outputs of these cases are off by at most
    rel 2.9e-3 and max 0.022 (attention over a cache), 0.04 (prefill), 0.1 (gradients): about four times that."""
    return {"rel": 1.2e-2, "max": 0.4 if case["path"] == "train" else 0.16 if case["path"] in ("prefill", "cold", "edit") else 0.09}
