"""The host side of the library's calls without a GPU: its objects linked with a stand-in for the
CUDA runtime (fake_cudart.cpp), which runs no kernel but follows what each stream is ordered after
and can make any call that queues work fail."""
import ctypes
import os
import re
import subprocess

import pytest

from paper_1904_03409_gb300 import build

HERE = os.path.dirname(os.path.abspath(__file__))
FP32, BF16 = 0, 1
USER = 0x77  # the caller's stream
SL_ERR_CUDA = 5


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    build.build()
    so = str(tmp_path_factory.mktemp("fake") / "libstacklstm_fake.so")
    include = os.path.join(os.path.dirname(os.path.dirname(build._nvcc())), "include")
    objs = [os.path.join(build.BUILD, os.path.basename(s)[:-3] + ".o") for s in build.sources()]
    subprocess.check_call(["g++", "-O1", "-std=c++17", "-fPIC", "-shared", "-Wl,-Bsymbolic", "-I" + include,
                           os.path.join(HERE, "fake_cudart.cpp"), *objs, "-lpthread", "-o", so])
    lib = ctypes.CDLL(so)
    vp = ctypes.c_void_p
    lib.fake_calls.restype = lib.fake_unjoined.restype = ctypes.c_long
    lib.fake_fail_at.argtypes = [ctypes.c_long]
    lib.fake_unjoined.argtypes = [vp]
    lib.fake_log.restype = lib.stacklstm_plan.restype = ctypes.c_char_p
    lib.stacklstm_create.argtypes = [ctypes.POINTER(vp)] + [ctypes.c_int] * 6 + [vp]
    lib.stacklstm_head_create.argtypes = [ctypes.POINTER(vp)] + [ctypes.c_int] * 7 + [vp]
    for name, n in (("forward", 13), ("backward", 8), ("plan", 1), ("destroy", 1), ("head_run", 21), ("head_destroy", 1)):
        getattr(lib, "stacklstm_" + name).argtypes = [vp] * n
    lib.stacklstm_set_async.argtypes = [vp, ctypes.c_int]
    return lib


class ForwardArgs(ctypes.Structure):  # sl_forward_args
    _fields_ = [("p%d" % i, ctypes.c_void_p) for i in range(12)]


class BackwardArgs(ctypes.Structure):  # sl_backward_args
    _fields_ = [("p%d" % i, ctypes.c_void_p) for i in range(7)]


def tensors(n):
    """n addresses of the caller's."""
    return [0x100000 * (i + 1) for i in range(n)]


def create(lib, T, B, I, H, dtype):
    h = ctypes.c_void_p()
    assert lib.stacklstm_create(ctypes.byref(h), T, B, I, H, dtype, 0, USER) == 0
    assert lib.stacklstm_set_async(h, 1) == 0
    return h


def forward(lib, h):
    return lib.stacklstm_forward(h, *tensors(12))


def backward(lib, h, d_top=True, dy=True):
    t = tensors(7)
    return lib.stacklstm_backward(h, t[0] if d_top else None, t[1] if dy else None, *t[2:])


def launches(lib):
    """(kernel, grid, block, shared memory, stream) of each launch."""
    out = []
    for line in lib.fake_log().decode().splitlines():
        f = line.split()
        out.append((f[0], tuple(map(int, f[1:4])), int(f[4]), int(f[5]), int(f[6])))
    return out


@pytest.mark.parametrize("T,B,I,H,dtype", [(20, 64, 200, 200, BF16), (20, 64, 75, 100, FP32), (6, 256, 64, 512, BF16),
                                           (4, 4, 16, 16, FP32)])
@pytest.mark.parametrize("what", ["forward", "backward"])
def test_a_call_that_fails_leaves_no_work_beside_the_callers_stream(lib, T, B, I, H, dtype, what):
    """Whichever call fails, what was queued on the handle's own stream and reads or writes the
    caller's tensors is waited for by the caller's stream (or the host) when the call returns.
    (The clear of the handle's own workspace is not: the next backward waits for it.)"""
    h = create(lib, T, B, I, H, dtype)

    def attempt(fail_at):
        lib.fake_reset()
        assert forward(lib, h) == 0
        if what == "forward":
            assert backward(lib, h) == 0
        lib.fake_reset()
        lib.fake_fail_at(fail_at)
        st = (forward if what == "forward" else backward)(lib, h)
        return st, lib.fake_calls(), lib.fake_unjoined(USER), launches(lib)

    st, n, left, log = attempt(-1)
    assert st == 0 and n > 8 and any(s != USER for *_, s in log)
    clears = left  # a complete forward: the clear alone
    assert clears <= (2 if what == "forward" else 0)
    for k in range(n):
        st, _, left, _ = attempt(k)
        assert st == SL_ERR_CUDA, (k, st)
        assert left <= clears, (k, left)
    lib.fake_reset()
    lib.stacklstm_destroy(h)


def test_a_head_run_that_fails_leaves_no_work_beside_the_callers_stream(lib):
    def attempt(fail_at):
        h = ctypes.c_void_p()
        assert lib.stacklstm_head_create(ctypes.byref(h), 19, 29, 8, 64, 64, 3, 0, USER) == 0
        lib.fake_reset()
        lib.fake_fail_at(fail_at)
        st = lib.stacklstm_head_run(h, *tensors(20))
        n, left = lib.fake_calls(), lib.fake_unjoined(USER)
        lib.stacklstm_head_destroy(h)
        lib.fake_reset()
        return st, n, left

    st, n, left = attempt(-1)
    assert st == 0 and left == 0 and n > 20
    for k in range(n):
        st, _, left = attempt(k)
        assert st == SL_ERR_CUDA, (k, st)
        assert left == 0, (k, left)


@pytest.mark.parametrize("T,kernel", [(1567, "seed_grads_dy_kernel"), (1568, "seed_grads_dy_kernel"),
                                      (1599, "seed_grads_dy_kernel"), (1600, "seed_grads_kernel")])
def test_per_step_seeding_keeps_its_rows_in_shared_memory_up_to_1599_steps(lib, T, kernel):
    h = create(lib, T, 4, 40, 40, BF16)
    assert forward(lib, h) == 0
    lib.fake_reset()
    assert backward(lib, h) == 0
    seeds = [l for l in launches(lib) if "seed_grads" in l[0]]
    lib.stacklstm_destroy(h)
    assert len(seeds) == 1 and kernel in seeds[0][0], seeds
    assert seeds[0][3] <= 227 * 1024


@pytest.mark.parametrize("B,H,dtype", [(65535, 32776, BF16), (3, 40, BF16), (3, 41, FP32)])
def test_initial_state_gradients_are_counted_beyond_32_bits(lib, B, H, dtype):
    """B x H past 2^31 elements: the launch that copies dh0 and dc0 has a grid of its size."""
    h = create(lib, 1, B, 8, H, dtype)
    assert forward(lib, h) == 0
    lib.fake_reset()
    assert backward(lib, h, dy=False) == 0
    copies = [l for l in launches(lib) if "h0_grads" in l[0]]
    lib.stacklstm_destroy(h)
    assert len(copies) == 1 and copies[0][1] == (min(152, -(-B * H // 256)), 1, 1), copies


@pytest.mark.parametrize("T,B,I,H,steps", [
    (1, 40, 33, 33, 1), (1, 8000, 64, 64, 1), (2, 8000, 64, 64, 0), (1, 128, 100, 100, 0), (1, 512, 100, 100, 1),
    (1, 1024, 200, 200, 0), (1, 4096, 200, 200, 1), (3, 4000, 16, 3, 3), (6, 4000, 16, 3, 0), (8, 40000, 16, 1, 8),
    (1, 40, 12300, 33, 0)])
def test_fp32_forward_of_few_steps_takes_the_step_kernel_where_it_is_shorter(lib, T, B, I, H, steps):
    """Beside a backward in row clusters; y then comes from the history like before them."""
    h = create(lib, T, B, I, H, FP32)
    assert b"clusters" in lib.stacklstm_plan(h)
    lib.fake_reset()
    assert forward(lib, h) == 0
    fwd = [l[0] for l in launches(lib)]
    lib.fake_reset()
    assert backward(lib, h) == 0
    bwd = [l[0] for l in launches(lib)]
    lib.stacklstm_destroy(h)
    assert sum("fwd_step_f32" in k for k in fwd) == steps, fwd
    assert sum("fwd_rows_f32" in k for k in fwd) == (0 if steps else 1), fwd
    assert sum("gather_rows" in k for k in fwd) == (3 if steps else 2), fwd  # h_stack, c_stack, y
    assert sum("bwd_rows_f32" in k for k in bwd) == 1, bwd


@pytest.mark.parametrize("H,dtype,lanes", [(1, FP32, 1), (8, BF16, 1), (16, BF16, 2), (24, BF16, 4), (9, FP32, 16),
                                           (64, FP32, 16), (136, BF16, 32), (33, FP32, 32), (104, FP32, 32)])
def test_gathers_give_a_row_no_more_lanes_than_it_has_pieces(lib, H, dtype, lanes):
    h = create(lib, 3, 1999, 8, H, dtype)
    lib.fake_reset()
    assert forward(lib, h) == 0
    gathers = [l for l in launches(lib) if "gather_rows" in l[0]]
    lib.stacklstm_destroy(h)
    # h_stack, before c_stack: four rows to each group of lanes, eight warps a block
    assert gathers[-2][1][0] == -(-4 * 1999 * lanes // 1024), gathers
    assert ("Lb1E" in gathers[-2][0]) == (lanes == 32), gathers


@pytest.mark.parametrize("B,I,early", [(64, 200, True), (64, 520, False), (8, 200, False), (200, 200, False)])
def test_the_clear_comes_before_the_steps_where_clusters_could_share_sms_without_need(lib, B, I, early):
    """Row clusters that fit two CTAs an SM and have an SM for each of several clusters' CTAs: the
    gradient history's clear is joined before the steps. One CTA an SM (a wide input), one cluster,
    or more clusters than that: it runs beside them, and the next backward waits for it."""
    h = create(lib, 40, B, I, 200, BF16)
    plan = lib.stacklstm_plan(h).decode()
    assert "rows 8" in plan and ("per SM %d rows" % (2 if I == 200 else 1)) in plan.split("; backward")[0], plan
    lib.fake_reset()
    assert forward(lib, h) == 0
    left = lib.fake_unjoined(USER)
    lib.stacklstm_destroy(h)
    assert left == (0 if early else 1)


@pytest.mark.parametrize("members,env,fwd,bwd", [
    # (B, I, H) of each: one launch of row clusters
    ([(64, 200, 200), (64, 48, 200), (1, 8, 208)], {}, 1, 1),
    # another contraction depth, more than 64 rows, clusters of other rows, an input too wide for them
    ([(64, 200, 208), (64, 200, 216)], {}, 2, 2),
    ([(64, 200, 200), (65, 200, 200)], {}, 2, 2),
    ([(64, 48, 200), (64, 680, 200)], {}, 2, 2),
    # wide inputs: the backward's 64-row clusters in one launch, persistent forwards
    ([(64, 680, 200), (9, 800, 200)], {}, 2, 1),
    # without row clusters the 64-row forwards, too, run one by one
    ([(64, 200, 200), (64, 48, 200)], {"STACKLSTM_ROW_CLUSTER": "0"}, 2, 1)])
def test_grouped_calls_share_a_launch_where_the_kernel_is_the_same(lib, monkeypatch, members, env, fwd, bwd):
    for k, v in env.items():
        monkeypatch.setenv(k, v)
    n = len(members)
    hs = [create(lib, 12, B, I, H, BF16) for B, I, H in members]
    handles = (ctypes.c_void_p * n)(*(h.value for h in hs))
    lib.fake_reset()
    assert lib.stacklstm_forward_group(n, handles, (ForwardArgs * n)(*[ForwardArgs(*tensors(12))] * n)) == 0
    steps = [l[0] for l in launches(lib) if "step_" in l[0]]
    assert len(steps) == fwd, steps
    lib.fake_reset()
    assert lib.stacklstm_backward_group(n, handles, (BackwardArgs * n)(*[BackwardArgs(*tensors(7))] * n)) == 0
    steps = [l[0] for l in launches(lib) if "step_" in l[0]]
    assert len(steps) == bwd, steps
    for h in hs:
        lib.stacklstm_destroy(h)


@pytest.mark.parametrize("T,H,dtype,units", [
    (60, 256, BF16, 4), (80, 256, BF16, 2), (256, 1024, BF16, 2), (270, 1024, BF16, 1), (60, 32, BF16, 1), (60, 64, BF16, 2),
    (60, 40, BF16, 2), (60, 104, BF16, 4), (60, 200, BF16, 1), (60, 8, BF16, 1), (60, 100, FP32, 4), (60, 66, FP32, 1),
    (60, 62, FP32, 2), (60, 63, FP32, 1)])
def test_per_step_seeding_leaves_no_lanes_idle_for_more_units_a_lane(lib, T, H, dtype, units):
    h = create(lib, T, 40, 8, H, dtype)
    assert forward(lib, h) == 0
    lib.fake_reset()
    assert backward(lib, h) == 0
    seeds = [l for l in launches(lib) if "seed_grads_dy" in l[0]]
    lib.stacklstm_destroy(h)
    assert len(seeds) == 1 and "ILi%dE" % units in seeds[0][0], seeds
    assert seeds[0][1] == (40, -(-H // (32 * units)), 1), seeds


def persistent_bytes(part, fwd, chunks):
    """What a persistent step kernel lays out in shared memory under its plan: alignment, a resident
    weight tile, the ring, the staging tile, a cluster's exchange tile, the barriers."""
    f = {k: int(v) for k, v in re.findall(r"(U|G|ring|w_res|smem|cluster|parts)[ =](\d+)", part.split(" dx CTAs")[0])}
    nb, ks = (4 * f["U"], 1) if fwd else (f["U"], f["parts"])
    weights = -(-chunks // ks) * nb * 128
    stage = f["G"] * (16384 + (0 if f["w_res"] else nb * 128))
    staging = 128 * f["U"] * 14 if fwd else 128 * 128 if f["U"] == 32 else 0
    exchange = 128 * f["U"] * 4 if f["cluster"] > 1 else 0
    return 1024 + f["w_res"] * weights + f["ring"] * stage + staging + exchange + 39 * 8 + 32, f["smem"]


@pytest.mark.parametrize("B", [8, 155, 300, 1000])
def test_persistent_plans_have_room_for_all_they_lay_out(lib, B):
    for H in [*range(264, 1040, 8), 1536, 2048]:
        h = create(lib, 5, B, 64, H, BF16)
        plan = lib.stacklstm_plan(h).decode()
        lib.stacklstm_destroy(h)
        fwd, bwd = plan.split("; step rings")[0].split("; backward ")
        chunks = re.search(r"chunks fwd (\d+) .*? bwd (\d+);", plan)
        for part, is_fwd, k in ((fwd.split("; forward ")[1], True, 1), (bwd, False, 2)):
            if part.startswith("persistent"):
                need, has = persistent_bytes(part, is_fwd, int(chunks.group(k)))
                assert need <= has <= 226 * 1024, (H, part)
