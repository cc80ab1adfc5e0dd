"""GPU parity of the clusters of 8 and 16 rows (bf16_rows.cu) against the fp64 oracle.

The shapes sit at the edges of their tiles: hidden widths that fill a warp's 8 units, a
CTA's 32 or an M tile's 16 exactly or partly, each contraction depth they are built for,
batches that leave rows of a group empty, one to three steps (fewer than the buffers in
flight), inputs wider than W_x's tiles, enough groups for two CTAs an SM, and more rows than
8-row groups fit. Outputs are
NaN-filled first; the 64-row clusters they replace run beside them.
"""
import os

import numpy as np
import pytest

import oracle
from paper_1904_03409_gb300 import binding as bd
from paper_1904_03409_gb300 import runner, workloads as wl
from parity import compare

pytestmark = pytest.mark.gpu


def plan_of(w):
    hd = bd.stacklstm_create(w.T, w.B, w.I, w.H, bd.SL_BF16, 0)
    try:
        return bd.stacklstm_plan(hd)
    finally:
        hd.destroy()


@pytest.mark.parametrize("T,B,I,H,seed", [
    (1, 2, 8, 8, 71), (2, 9, 8, 32, 72), (3, 8, 24, 64, 73), (5, 17, 208, 72, 74), (6, 5, 40, 128, 75),
    (50, 1, 40, 200, 76), (7, 12, 16, 208, 77), (4, 3, 72, 216, 78), (9, 10, 256, 256, 79), (6, 20, 520, 104, 80),
    (4, 250, 16, 200, 81), (4, 500, 16, 200, 83), (3, 573, 200, 176, 84), (2, 561, 24, 136, 85)])
def test_row_clusters_match_oracle(T, B, I, H, seed):
    w = wl.make_workload("case", T=T, B=B, I=I, H=H, dtype="bf16", seed=seed, ops_kind="random_walk",
                         probs=(0.5, 0.3, 0.2), bias_scale=0.3, h0_scale=0.5, c0_scale=0.5, dy_scale=0.5)
    rows = "rows 16" if B > 288 else "rows 8"
    assert plan_of(w).count(rows) == 2, plan_of(w)
    args = (w.x, w.ops, w.h0, w.c0, w.W, w.bias)
    ref = oracle.run(*args, d_top_h=w.d_top_h, dy=w.dy)
    got = runner.run(w)
    compare(got, ref, "bf16")
    again = runner.run(w)
    for k in ("y", "h_stack", "c_stack", "dx", "dW", "dbias", "dh0", "dc0"):
        assert np.array_equal(got[k], again[k]), k
    compare(runner.run(w, mode=bd.SL_MODE_PUSH_ONLY),
            oracle.run(*args, d_top_h=w.d_top_h, dy=w.dy, mode="definition"), "bf16")
    os.environ["STACKLSTM_ROW_CLUSTER"] = "0"
    try:
        assert rows not in plan_of(w)
        compare(runner.run(w), ref, "bf16")
    finally:
        del os.environ["STACKLSTM_ROW_CLUSTER"]


def test_final_top_gradient_without_dy():
    """The loss on the final tops alone: the backward launch adds it itself."""
    w = wl.make_workload("case", T=20, B=21, I=16, H=40, dtype="bf16", seed=82, ops_kind="random_walk",
                         probs=(0.5, 0.3, 0.2), bias_scale=0.3, h0_scale=0.5)
    for mode, name in ((bd.SL_MODE_HOMOGENIZED, "homogenized"), (bd.SL_MODE_PUSH_ONLY, "definition")):
        compare(runner.run(w, mode=mode), oracle.run(w.x, w.ops, w.h0, w.c0, w.W, w.bias, d_top_h=w.d_top_h, mode=name),
                "bf16")
