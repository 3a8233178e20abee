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
