"""GPU parity of the fp32 CUDA-core path against the fp64 oracle, and the device-side
error statuses. Runs through the C ABI on cuda:0."""
import numpy as np
import pytest
import torch

import oracle
from paper_1904_03409_gb300 import binding as bd
from paper_1904_03409_gb300 import runner, workloads as wl
from parity import compare

pytestmark = pytest.mark.gpu


def oracle_of(w, d_top_h=None):
    return oracle.run(w.x, w.ops, w.h0, w.c0, w.W, w.bias, d_top_h=w.d_top_h if d_top_h is None else d_top_h,
                      dy=w.dy)


def test_tiny_config():
    w = wl.config_workload("tiny")
    got = runner.run(w)
    compare(got, oracle_of(w), "fp32")


@pytest.mark.parametrize("T,B,I,H,seed,probs", [
    (33, 37, 24, 40, 1, (0.5, 0.3, 0.2)),    # ragged B, H not a multiple of 32
    (50, 5, 7, 33, 2, (0.4, 0.4, 0.2)),      # odd sizes
    (20, 130, 16, 160, 3, (0.6, 0.3, 0.1)),  # several thread blocks per instance
    (1, 3, 4, 5, 4, (1.0, 0.0, 0.0)),        # a single step
])
def test_random_cases(T, B, I, H, seed, probs):
    w = wl.make_workload("case", T=T, B=B, I=I, H=H, dtype="fp32", seed=seed, ops_kind="random_walk",
                         probs=probs, bias_scale=0.3, h0_scale=0.5, c0_scale=0.5, dy_scale=0.5)
    got = runner.run(w)
    compare(got, oracle_of(w), "fp32")


@pytest.mark.parametrize("T,B,I,H,seed", [(12, 4, 16, 16, 10), (20, 16, 16, 32, 11), (9, 20, 8, 48, 12)])
def test_one_cta_and_per_step_kernels_agree_bit_for_bit(T, B, I, H, seed):
    """Small problems run each direction's steps in one CTA; the per-step kernels
    (STACKLSTM_STEP_KERNELS=1) do the same arithmetic per element, so every output is
    bit-identical, and both match the oracle."""
    import os
    w = wl.make_workload("case", T=T, B=B, I=I, H=H, dtype="fp32", seed=seed, ops_kind="random_walk",
                         probs=(0.5, 0.3, 0.2), bias_scale=0.3, h0_scale=0.5, c0_scale=0.5, dy_scale=0.5)
    hd = bd.stacklstm_create(T, B, I, H, bd.SL_FP32, 0)
    try:
        assert "one CTA" in bd.stacklstm_plan(hd)
    finally:
        hd.destroy()
    one = runner.run(w)
    os.environ["STACKLSTM_STEP_KERNELS"] = "1"
    try:
        hd = bd.stacklstm_create(T, B, I, H, bd.SL_FP32, 0)
        try:
            assert "one launch per step" in bd.stacklstm_plan(hd)
        finally:
            hd.destroy()
        per = runner.run(w)
    finally:
        os.environ.pop("STACKLSTM_STEP_KERNELS", None)
    for k in ("y", "h_stack", "c_stack", "dx", "dW", "dbias", "dh0", "dc0"):
        assert np.array_equal(one[k], per[k], equal_nan=False), k
    compare(one, oracle_of(w), "fp32")


def test_holds_only_and_all_push():
    for probs in ((0.0, 0.0, 1.0), (1.0, 0.0, 0.0)):
        w = wl.make_workload("case", T=16, B=9, I=8, H=12, dtype="fp32", seed=7, ops_kind="random_walk",
                             probs=probs, h0_scale=0.5)
        got = runner.run(w)
        compare(got, oracle_of(w), "fp32")
        if probs[2] == 1.0:
            assert np.all(got["dx"] == 0.0) and np.all(got["dW"] == 0.0)


def test_dead_writes_have_exactly_zero_input_gradient():
    w = wl.make_workload("case", T=40, B=16, I=8, H=12, dtype="fp32", seed=8, ops_kind="random_walk",
                         probs=(0.4, 0.4, 0.2))
    got = runner.run(w)
    assert np.all(got["dx"][w.ops != 1] == 0.0)


def test_backward_is_bitwise_reproducible():
    w = wl.make_workload("case", T=25, B=20, I=8, H=16, dtype="fp32", seed=9, ops_kind="random_walk",
                         probs=(0.5, 0.3, 0.2), dy_scale=1.0)
    a, b = runner.run(w), runner.run(w)
    for k in ("dx", "dW", "dbias", "dh0", "dc0"):
        assert np.array_equal(a[k], b[k]), k


def _statuses(ops_np):
    T, B = ops_np.shape
    hd = bd.stacklstm_create(T, B, 4, 4, bd.SL_FP32, 0)
    dev = torch.device("cuda", 0)
    z = lambda *s: torch.zeros(*s, device=dev)
    ops = torch.from_numpy(ops_np.astype(np.int8)).to(dev)
    pf = torch.zeros(B, dtype=torch.int32, device=dev)
    try:
        with pytest.raises(bd.StackLSTMError) as e:
            bd.stacklstm_forward(hd, z(T, B, 4), ops, z(B, 4), z(B, 4), z(8, 16), z(16), p_final=pf)
        return e.value.status, hd
    except BaseException:
        hd.destroy()
        raise


def test_bad_op_and_underflow_statuses():
    st, hd = _statuses(np.array([[1, 2], [0, 0]]))
    hd.destroy()
    assert st == 2
    st, hd = _statuses(np.array([[1, 0], [-1, -1]]))
    assert st == 3
    # the handle stays usable: a valid stream now succeeds
    dev = torch.device("cuda", 0)
    z = lambda *s: torch.zeros(*s, device=dev)
    pf = torch.zeros(2, dtype=torch.int32, device=dev)
    bd.stacklstm_forward(hd, z(2, 2, 4), torch.ones(2, 2, dtype=torch.int8, device=dev), z(2, 4), z(2, 4),
                         z(8, 16), z(16), p_final=pf)
    assert pf.tolist() == [2, 2]
    hd.destroy()


def test_backward_before_forward():
    hd = bd.stacklstm_create(3, 2, 4, 4, bd.SL_FP32, 0)
    try:
        with pytest.raises(bd.StackLSTMError) as e:
            bd.stacklstm_backward(hd)
        assert e.value.status == 4
    finally:
        hd.destroy()


@pytest.mark.parametrize("T,B,I,H,seed", [
    (5, 400, 7, 3, 21), (3, 41, 9, 33, 22), (2, 9, 17, 129, 23), (1, 70, 40, 200, 24), (40, 64, 200, 200, 25),
    (6, 5, 5, 225, 26), (4, 6, 130, 256, 27), (60, 13, 75, 100, 28), (30, 33, 1, 32, 29), (7, 90, 64, 177, 30),
    (500, 1, 11, 65, 31), (9, 300, 33, 64, 32)])
def test_row_clusters_match_oracle(T, B, I, H, seed):
    """Clusters of few rows (fp32_rows.cu): units that fill a warp's four or not, one CTA to
    eight, one row to eight a cluster with the last group partly empty, several rounds of
    clusters, one to three steps (fewer than the buffers in flight), sizes that divide no tile
    of the contractions, into NaN-filled outputs; reruns agree bit for bit."""
    w = wl.make_workload("case", T=T, B=B, I=I, H=H, dtype="fp32", seed=seed, ops_kind="random_walk",
                         probs=(0.5, 0.3, 0.2), bias_scale=0.3, h0_scale=0.5, c0_scale=0.5, dy_scale=0.5)
    hd = bd.stacklstm_create(T, B, I, H, bd.SL_FP32, 0)
    try:
        assert "clusters" in bd.stacklstm_plan(hd), bd.stacklstm_plan(hd)
    finally:
        hd.destroy()
    got = runner.run(w)
    compare(got, oracle_of(w), "fp32")
    again = runner.run(w)
    for k in ("y", "h_stack", "c_stack", "dx", "dW", "dbias", "dh0", "dc0"):
        assert np.array_equal(got[k], again[k]), k


@pytest.mark.parametrize("which", ["STACKLSTM_WAIT_LIMIT_CYCLES", "STACKLSTM_WAIT_LIMIT_BWD_CYCLES"])
def test_row_clusters_report_a_wait_that_runs_out(which):
    """With a zero wait limit (both directions, or the backward's) the call reports
    SL_ERR_TIMEOUT and the device stays usable."""
    import os
    w = wl.make_workload("case", T=12, B=64, I=16, H=120, dtype="fp32", seed=33, ops_kind="random_walk",
                         probs=(0.5, 0.3, 0.2))
    os.environ[which] = "0"
    try:
        hd = bd.stacklstm_create(w.T, w.B, w.I, w.H, bd.SL_FP32, 0)
    finally:
        del os.environ[which]
    try:
        assert "clusters" in bd.stacklstm_plan(hd)
        ins, out = runner.upload(w), runner.alloc_outputs(w)
        with pytest.raises(bd.StackLSTMError) as e:
            runner.forward_backward(hd, ins, out)
        assert e.value.status == 6
    finally:
        hd.destroy()
    compare(runner.run(w), oracle_of(w), "fp32")


@pytest.mark.parametrize("T,B,I,H", [(30, 33, 31, 32), (30, 33, 32, 32), (40, 47, 60, 67), (30, 50, 128, 128),
                                     (60, 64, 64, 256)])
def test_weight_and_bias_gradients_alone_equal_both(T, B, I, H):
    """dbias is a row of ones below the weight gradient's operand: alone, and dW alone, they are
    what the call that returns both gives, at row counts on both sides of a tile."""
    w = wl.make_workload("case", T=T, B=B, I=I, H=H, dtype="fp32", seed=41, ops_kind="random_walk",
                         probs=(0.5, 0.3, 0.2), bias_scale=0.3, h0_scale=0.5, c0_scale=0.5, dy_scale=0.5)
    hd = bd.stacklstm_create(T, B, I, H, bd.SL_FP32, 0)
    try:
        assert "clusters" in bd.stacklstm_plan(hd)
        ins, out = runner.upload(w), runner.alloc_outputs(w)
        runner.forward_backward(hd, ins, out)
        both = runner.to_numpy(out)
        compare(both, oracle_of(w), "fp32")
        for k in ("dW", "dbias"):
            part = runner.alloc_outputs(w)
            full = dict(part, **{{"dW": "dbias", "dbias": "dW"}[k]: None})
            runner.forward_backward(hd, ins, full)
            assert np.array_equal(full[k].cpu().numpy(), both[k]), k
    finally:
        hd.destroy()


@pytest.mark.parametrize("T,B,H", [(1, 1100, 8), (1, 60000, 8), (37, 320, 12), (1, 9001, 9), (185, 64, 40)])
def test_weight_gradient_sums_are_compensated(T, B, H):
    """The sums over all T B rows alone, their operands taken as they are. With I = 4H and the
    identity as W_x, dx is dG exactly; x and the states read (h0 at T = 1) are the other operand.
    Rounding the result alone leaves up to 2^-24 / sqrt(3) = 3.4e-8 in the 2-norm, and the products
    (two roundings of 2^-24 of a term at most, over n terms of like size) less than that; sums
    with rounding errors that add up over the rows of a split have 1.2e-7 and more."""
    I = 4 * H
    g = torch.Generator(device="cuda").manual_seed(T * B + H)
    r = lambda *s: torch.randn(*s, generator=g, device="cuda")
    W = torch.cat([torch.eye(I, device="cuda"), 0.1 * r(H, I)])
    ins = dict(x=r(T, B, I), ops=torch.ones(T, B, dtype=torch.int8, device="cuda"), h0=r(B, H), c0=r(B, H), W=W, bias=r(I))
    e = lambda *s: torch.full(s, float("nan"), device="cuda")
    y, dx, dh0, dc0, dW, dbias = e(T, B, H), e(T, B, I), e(B, H), e(B, H), e(I + H, I), e(I)
    hd = bd.stacklstm_create(T, B, I, H, bd.SL_FP32, 0)
    try:
        assert "clusters" in bd.stacklstm_plan(hd), bd.stacklstm_plan(hd)
        bd.stacklstm_forward(hd, *(ins[k] for k in ("x", "ops", "h0", "c0", "W", "bias")),
                             p_final=torch.empty(B, dtype=torch.int32, device="cuda"), y=y)
        bd.stacklstm_backward(hd, None, r(T, B, H), dx, dh0, dc0, dW, dbias)
    finally:
        hd.destroy()
    dG = dx.double().view(-1, I)
    read = torch.cat([ins["h0"][None], y[:-1]]).double().view(-1, H)  # pushes only: the step before's output
    rows = torch.cat([ins["x"].double().view(-1, I), read], 1)
    for got, want in ((dW, rows.t() @ dG), (dbias, dG.sum(0))):
        err = ((got.double() - want).norm() / want.norm()).item()
        assert err < 5e-8, err


@pytest.mark.parametrize("T,B,I,H,seed", [(1, 70, 40, 64, 51), (1, 300, 9, 33, 52), (1, 600, 16, 100, 53),
                                          (1, 513, 17, 99, 54), (3, 4100, 5, 3, 55), (2, 9000, 4, 1, 56),
                                          (1, 4097, 8, 132, 57)])
def test_step_forward_beside_the_row_clusters_backward(T, B, I, H, seed):
    """Forwards of one step, or of few at H <= 3, by the step kernel, and the backward in clusters:
    the weight gradient reads the rows [x ; h_read] that the step kernel kept, with and without
    the alignment for 16-byte copies; an output is the top's row of the history."""
    w = wl.make_workload("case", T=T, B=B, I=I, H=H, dtype="fp32", seed=seed, ops_kind="random_walk",
                         probs=(0.5, 0.3, 0.2), bias_scale=0.3, h0_scale=0.5, c0_scale=0.5, dy_scale=0.5)
    got = runner.run(w)
    compare(got, oracle_of(w), "fp32")
    again = runner.run(w)
    for k in ("y", "h_stack", "c_stack", "dx", "dW", "dbias", "dh0", "dc0"):
        assert np.array_equal(got[k], again[k]), k
