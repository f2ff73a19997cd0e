"""Buckets of a few tiles per SM: which kernel a fused step runs on, on both sides of the lines (148 SMs, tiles of 2048
elements), and that the kernels on either side of a line give the same state, bit for bit."""
import pytest
import torch

import paper_2507_07114_b200 as L
import workload
from parity_util import GpuRun, assert_rel, assert_same, to_np

pytestmark = pytest.mark.gpu
SM_TILE = 148 * 2048
# W, n, P, p, gradients, replicas, optimizer, start of the build's name
CASES = [
    (8, SM_TILE // 8 - 256, 256, 0.1, "bf16", "bf16", "adam", "gather wide"),        # under an eighth of a tile per SM
    (8, SM_TILE // 8 + 256, 256, 0.1, "bf16", "bf16", "adam", "register"),
    (3, 2 * SM_TILE - 512, 512, 0.3, "bf16", "bf16", "sgd", "register"),              # up to two, bf16 replicas
    (3, 2 * SM_TILE, 512, 0.3, "bf16", "bf16", "sgd", "gather twin"),
    (16, 2 * SM_TILE - 256 + 40, 256, 0.05, "bf16", "bf16", "adam", "register"),      # a short last packet
    (9, SM_TILE - 256, 256, 0.2, "f32", "f32", "adam", "register"),                   # up to one, fp32 replicas
    (9, SM_TILE, 256, 0.2, "f32", "f32", "adam", "gather wide"),
    (9, SM_TILE // 2, 512, 0.2, "f32", "f32", "adam", "gather wide"),                 # 512 elements: up to eight workers
    (8, SM_TILE // 2, 512, 0.2, "f32", "f32", "adam", "register"),
    (5, SM_TILE, 128, 0.1, "bf16", "bf16", "adam", "gather"),                         # 128 elements: never
    (8, 5 * SM_TILE - 736, 736, 0.1, "bf16", "bf16", "adam", "register"),             # chunks filled to 0.96: from eight tiles,
    (8, 8 * SM_TILE, 736, 0.1, "bf16", "bf16", "adam", "gather wide"),
    (6, 7 * SM_TILE // 2 + 136, 136, 0.1, "bf16", "bf16", "adam", "gather twin"),     # to 0.53: from three and a half,
    (6, 7 * SM_TILE // 2 - 136, 136, 0.1, "bf16", "bf16", "sgd", "register"),         # more for SGD
    (17, 4 * SM_TILE, 136, 0.1, "bf16", "bf16", "adam", "register"),                  # and many workers
]
# a short last packet behind packets from 1024 elements: one launch, up to the line
ONE_LAUNCH = [
    (4, 100_003, 1024, 0.1, "f32", "f32", "sgd", "register"),
    (9, 100_003, 1024, 0.1, "f32", "f32", "sgd", "bulk-copy twin"),                   # fp32 replicas: eight workers
    (8, 2 * SM_TILE + 9, 2048, 0.1, "bf16", "f32", "adam", "bulk-copy wide"),         # and two tiles per SM
    (8, SM_TILE // 8 - 3, 2048, 0.1, "f32", "f32", "adam", "bulk-copy wide"),         # from an eighth
    (8, SM_TILE // 8 + 3, 2048, 0.1, "f32", "f32", "adam", "register"),
    (8, SM_TILE - 5, 2048, 0.1, "bf16", "bf16", "adam", "bulk-copy wide"),            # bf16 replicas: from one
    (8, SM_TILE + 5, 2048, 0.1, "bf16", "bf16", "adam", "register"),
    (33, 3 * SM_TILE + 77, 2048, 0.2, "bf16", "bf16", "adam", "register"),            # to 3.6
    (14, 4 * SM_TILE + 5, 1024, 0.05, "bf16", "bf16", "adam", "bulk-copy wide group=8 stale=late packed"),
    (16, SM_TILE + 1000, 4480, 0.3, "bf16", "bf16", "adam", "register"),              # no multiple of 1024: to two
    (17, 2 * SM_TILE + 1000, 4480, 0.3, "bf16", "bf16", "adam", "bulk-copy twin"),
]


@pytest.mark.parametrize("case", CASES + ONE_LAUNCH, ids=["W%d-n%d-P%d-%s-%s" % (c[0], c[1], c[2], c[5], c[6]) for c in CASES + ONE_LAUNCH])
def test_small_buckets(case):
    W, n, P, p, g, r, opt, plan = case
    w = workload.Workload("small", W, n, P, p, opt, 3e-4, g, r, 2, seed=n % 97)
    a = GpuRun(w)
    got = L.lossy_describe_plan(a.ctx)
    assert got.startswith(plan), got
    other, flag = ("register", L.LOSSY_REGISTER_PATH) if plan != "register" else ("bulk-copy", L.LOSSY_PACKED_BULK) if case in ONE_LAUNCH else ("gather", L.LOSSY_GATHER_PATH)
    b = GpuRun(w, flags=flag)
    assert L.lossy_describe_plan(b.ctx).startswith(other)
    for t in (1, 2):
        grads = [workload.grad_slab(w, t, i, 0, n, "cuda") for i in range(W)]
        a.step_fused(t, grads)
        b.step_fused(t, grads)
    oa, ob = a.outputs(), b.outputs()
    for k in ("ghat", "count", "recv_bits", "stale_bits"):
        assert_same(oa[k], ob[k], k)
    assert_rel(oa["sumsq"], ob["sumsq"], "drift sums", tol=1e-7)     # fp32 squares summed in other trees: 1e-8
    for name in ("master", "m", "v"):
        assert_same(to_np(getattr(a, name)), to_np(getattr(b, name)), name)
    for i in range(W):
        assert torch.equal(a.replicas[i], b.replicas[i]), f"replica {i}"
    L.lossy_device_status(a.ctx)
    L.lossy_device_status(b.ctx)


# W, n, P, gradients, replicas, start of the build's name without drift norms, and with
NO_NORMS = [(32, SM_TILE // 2, 256, "f32", "f32", "gather wide", "register"),
            (24, SM_TILE // 2, 256, "f32", "f32", "register", "register"),
            (32, SM_TILE // 2, 256, "bf16", "bf16", "register", "register"),
            (25, SM_TILE - 256 + 40, 256, "bf16", "f32", "gather wide", "register"),      # a short last packet
            (8, SM_TILE, 2048, "bf16", "bf16", "bulk-copy wide", "bulk-copy wide"),
            (8, SM_TILE + 5, 2048, "bf16", "bf16", "bulk-copy wide", "register")]


@pytest.mark.parametrize("W,n,P,g,r,without,with_norms", NO_NORMS)
def test_small_buckets_without_drift_norms(W, n, P, g, r, without, with_norms):
    w = workload.Workload("no_norms", W, n, P, 0.1, "adam", 3e-4, g, r, 2, seed=n % 97)
    a, b = GpuRun(w), GpuRun(w)
    assert L.lossy_describe_plan(a.ctx, with_drift=False).startswith(without)
    assert L.lossy_describe_plan(b.ctx).startswith(with_norms)
    grads = [workload.grad_slab(w, 1, i, 0, n, "cuda") for i in range(W)]
    for t in (1, 2):
        L.lossy_fused_step(a.ctx, t, grads, a.master, a.m, a.v, a.replicas, a.ghat, a.count, a.recv, a.stale)
        b.step_fused(t, grads)
    oa, ob = a.outputs(), b.outputs()
    for k in ("ghat", "count", "recv_bits", "stale_bits"):
        assert_same(oa[k], ob[k], k)
    for name in ("master", "m", "v"):
        assert_same(to_np(getattr(a, name)), to_np(getattr(b, name)), name)
    for i in range(W):
        assert torch.equal(a.replicas[i], b.replicas[i]), f"replica {i}"
    L.lossy_device_status(a.ctx)
