"""The planning arithmetic of the attention launches (csrc/ba_plan.h, plain C++): every plan that a launch could be made from covers
every key tile of every item exactly once and stays within its room for partial results.  What a CTA of a plan does is stated
here from the launches' definitions, with the closed forms the kernels use."""
import ctypes as C
import os
import shutil
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SNAP = 2                                                     # a cut this close to an item's edge moves to the edge

SOURCE = r"""
#include "ba_plan.h"
extern "C" void stream_plan(int sms, int chunks, const int32_t *tiles, int odd, int cap, long long *out) {
  const ba_stream_plan p = ba_plan_stream(sms, chunks, tiles, odd, cap);
  out[0] = p.n_ctas; out[1] = p.n_odd; out[2] = p.n_slots; out[3] = p.cost;
}
extern "C" void cluster_plan(long long items, int two, int one, int fused, long long tiles, const int32_t *at_a_time, double *out) {
  const ba_cluster_plan p = ba_plan_cluster(items, two != 0, one != 0, fused != 0, tiles, [&](int n) { return at_a_time[n]; });
  out[0] = p.size; out[1] = p.single; out[2] = p.cost; out[3] = p.shared;
}
extern "C" int final_splits(int sms, int chunks, int items, int tiles, int longest, int cap) {
  return ba_plan_final_splits(sms, chunks, items, tiles, longest, cap);
}
"""


@pytest.fixture(scope="module")
def plans(tmp_path_factory):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no C++ compiler")
    d = tmp_path_factory.mktemp("plans")
    (d / "plans.cc").write_text(SOURCE)
    subprocess.run([gxx, "-std=c++17", "-shared", "-fPIC", "-I", os.path.join(ROOT, "paper_2409_15355_b200", "csrc"), str(d / "plans.cc"),
                    "-o", str(d / "plans.so")], check=True)
    lib = C.CDLL(str(d / "plans.so"))
    lib.cluster_plan.argtypes = [C.c_longlong, C.c_int, C.c_int, C.c_int, C.c_longlong, C.POINTER(C.c_int32 * 9), C.POINTER(C.c_double * 4)]
    return lib


def _stream_plan(plans, sms, chunks, sequences, cap):
    items = [n for seq in sequences for n in seq]
    odd = sum(n for seq in sequences for n in seq[1::2])
    out = (C.c_longlong * 4)()
    plans.stream_plan(sms, chunks, (C.c_int32 * 3)(sum(items), min(items), max(items)), odd, cap, out)
    return tuple(out)


def _check_stream(sequences, chunks, n_ctas, n_odd, n_slots):
    """sequences: key tiles of the items of every sequence.  Items 0, 2, .. of all (sequence, chunk) lie end to end in one stream, items
    1, 3, .. in another, on the last n_odd of the CTAs; each stream is cut into one run per CTA."""
    taken, slots = {}, {}
    for lane, g in ((0, n_ctas - n_odd), (1, n_odd)):
        line, at = [], 0                                     # (key, first tile, tiles) of the items in stream order
        for s, seq in enumerate(sequences):
            for c in range(chunks):
                for i in range(lane, len(seq), 2):
                    line.append(((s, c, i), at, seq[i]))
                    at += seq[i]
        total = at
        if total == 0:
            assert g == 0
            continue
        assert g > 0, "a stream that no CTA takes"

        def moved(x):
            for _, g0, n in line:
                if g0 <= x < g0 + n:
                    return g0 if x - g0 <= SNAP else g0 + n if g0 + n - x <= SNAP else x
            return x
        cuts = [moved(total * j // g) for j in range(g + 1)]
        assert cuts[0] == 0 and cuts[-1] == total and cuts == sorted(cuts)
        for cta in range(g):
            for key, g0, n in line:
                a, b = max(cuts[cta], g0), min(cuts[cta + 1], g0 + n)
                if a >= b:
                    continue
                taken.setdefault(key, []).extend(range(a - g0, b - g0))
                last = lambda x: min(g - 1, ((x + 1) * g - 1) // total)   # noqa: E731  the last CTA whose raw cut is at most x
                j0 = last(g0 + min(SNAP, n - 1))
                j1 = max(j0, last(g0 + n - SNAP - 1))
                assert j0 <= cta <= j1
                if j1 > j0:
                    assert j1 - j0 < n_slots
                    slots.setdefault(key, {})[cta - j0] = cta == j1      # the last piece marks the slots behind it empty
                else:
                    assert (a, b) == (g0, g0 + n)                          # a whole item, written without partial results
    for s, seq in enumerate(sequences):
        for c in range(chunks):
            for i, n in enumerate(seq):
                assert sorted(taken.get((s, c, i), [])) == list(range(n)), (s, c, i)
    for used in slots.values():
        top = max(used)
        assert sorted(used) == list(range(top + 1)) and used[top] and not any(used[k] for k in range(top))


def _item_lists(rng):
    """Key tiles of the items of a few sequences: cached tiles and one more own tile every one or two items."""
    sequences = []
    for _ in range(int(rng.integers(1, rng.choice([2, 3, 8, 40])))):
        cached, n, step = int(rng.integers(0, rng.choice([1, 3, 20, 90]))), int(rng.integers(1, rng.choice([2, 3, 6]))), int(rng.integers(1, 3))
        sequences.append([cached + 1 + i // step for i in range(n)])
    return sequences


def test_every_stream_plan_covers_every_tile_once(plans):
    rng = np.random.default_rng(11)
    planned = 0
    for _ in range(4000):
        sms, chunks, cap = int(rng.choice([1, 2, 7, 20])), int(rng.choice([1, 1, 2, 3])), int(rng.integers(1, 33))
        sequences = _item_lists(rng)
        n_ctas, n_odd, n_slots, _ = _stream_plan(plans, sms, chunks, sequences, cap)
        if n_ctas == 0:
            continue
        planned += 1
        assert 0 <= n_odd < n_ctas <= sms and 1 <= n_slots <= cap
        _check_stream(sequences, chunks, n_ctas, n_odd, n_slots)
    assert planned > 1000


@pytest.mark.parametrize("sequences", [[[1, 1]], [[1], [1]], [[1, 1], [1]], [[2, 2]], [[1, 1, 1]], [[3, 3]]], ids=str)
@pytest.mark.parametrize("sms", [1, 2, 3, 148])
def test_stream_plans_of_the_smallest_lists(plans, sequences, sms):
    n_ctas, n_odd, n_slots, _ = _stream_plan(plans, sms, 1, sequences, 32)
    if n_ctas:
        _check_stream(sequences, 1, n_ctas, n_odd, n_slots)


def test_stream_plan_of_a_serving_batch(plans):
    """Sixteen requests of 53 and 54 tiles, eight chunks: one run per SM, runs within a tile of one another."""
    sequences = [[53, 54]] * 16
    n_ctas, n_odd, n_slots, cost = _stream_plan(plans, 148, 8, sequences, 32)
    assert n_ctas == 148 and 60 < n_odd < 90 and n_slots <= 4
    _check_stream(sequences, 8, n_ctas, n_odd, n_slots)
    assert cost < 107 * 16 * 8 // 148 + 20


def test_cluster_plans_take_the_cheapest_size_that_fits(plans):
    rng = np.random.default_rng(12)
    chosen = 0
    for _ in range(3000):
        items, two, tiles = int(rng.integers(1, 200)), bool(rng.integers(2)), int(rng.integers(1, 120))
        fits = (C.c_int32 * 9)(*[0, 0] + [int(rng.choice([0, 148 // n])) for n in range(2, 9)])
        out = (C.c_double * 4)()
        one = not two and bool(rng.integers(2))                           # (two: on average more than one query tile an item)
        fused = bool(rng.integers(2))
        plans.cluster_plan(items, two, one, fused, tiles, C.byref(fits), C.byref(out))
        size, single, cost, shared = int(out[0]), int(out[1]), out[2], int(out[3])
        want = {}
        for s in (0, 1)[:2 if two else 1]:
            for n in range(2, min(8, tiles) + 1):
                units = items << s
                if units > 1 and fits[n] < 1:
                    continue
                rounds = -(-units // (1 if units == 1 else fits[n]))
                tile, start, merge = (0.6, 3.5, 0.25) if not fused and (s or one) else (0.85, 3, 0.25) if s else (1.0, 3, 1.5)
                want[n, s] = rounds * (-(-tiles // n) * tile + start) + merge
        if not want:
            assert size == 0 and not shared
            continue
        chosen += 1
        assert shared == (not fused and (single or one))                 # a CTA with two query tiles: the kernel without sharing
        assert 2 <= size <= min(8, tiles) and (not single or two)
        assert cost == pytest.approx(min(want.values())) and want[size, single] == pytest.approx(cost)
        cuts = [tiles * k // size for k in range(size + 1)]                # every CTA has a share, none is empty
        assert cuts[0] == 0 and cuts[-1] == tiles and all(b > a for a, b in zip(cuts, cuts[1:]))
    assert chosen > 2000


# Shapes whose layouts were all timed: items, more than one query tile an item, all of one, key tiles, the fastest (size, single) and the
# price of the best layout without a cluster.  148 SMs, clusters at a time as the driver gives them.
@pytest.mark.parametrize("items,two,one,tiles,best,without", [(16, True, False, 48, (4, 1), 14), (32, True, False, 9, (2, 1), 11),
                                                              (8, True, False, 48, (6, 1), 11), (16, False, True, 71, (6, 0), 16)])
def test_cluster_plans_where_every_layout_was_timed(plans, items, two, one, tiles, best, without):
    fits, out = (C.c_int32 * 9)(0, 0, 74, 45, 33, 26, 22, 15, 15), (C.c_double * 4)()
    plans.cluster_plan(items, two, one, 0, tiles, C.byref(fits), C.byref(out))
    assert (int(out[0]), int(out[1])) == best and out[3] == 1 and out[2] < without


def test_final_blocks_of_a_prefill_are_cut_only_where_they_would_end_the_launch(plans):
    rng = np.random.default_rng(13)
    cut = 0
    for _ in range(3000):
        sms, chunks, items = int(rng.choice([20, 148])), int(rng.choice([1, 2, 8])), int(rng.integers(1, 400))
        longest = int(rng.integers(1, 300))
        tiles, cap = longest + int(rng.integers(0, 6)) * items, int(rng.integers(0, 17))
        n = plans.final_splits(sms, chunks, items, tiles, longest, cap)
        assert 1 <= n <= max(1, cap)
        share = (tiles + items) * chunks // sms
        if longest <= max(share // 2, 6):
            assert n == 1
        elif cap >= 2:
            cut += 1
            assert n == cap or -(-longest // n) <= max(share // 2, 6)
    assert cut > 500
