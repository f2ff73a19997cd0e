"""Kernels begin while the kernel ahead of them in the stream still runs and wait for its end themselves, and the launch
of a short last packet runs beside the launch of the complete ones. So calls issued without a pause, of several buckets on
one stream and inside a captured graph, must give the bits that calls with a synchronisation after each give."""
import pytest
import torch

import paper_2507_07114_b200 as L
import workload
from parity_util import GpuRun, assert_same, to_np

pytestmark = pytest.mark.gpu

# W, n, P, p, optimizer, types, mode, start of the build's name: each with a short last packet, on every kernel that a fused step runs
# on. All but the register kernel's buckets take two launches.
BUCKETS = [(4, 1024 * 700 + 675, 1024, 0.1, "sgd", "f32", "f32", "", "bulk-copy twin"),
           (8, 2048 * 550 + 3, 2048, 0.1, "adam", "bf16", "bf16", "", "bulk-copy wide"),     # a last packet of three elements
           (12, 256 * 4000 + 40, 256, 0.1, "adam", "bf16", "bf16", "", "gather wide"),
           (3, 320 * 50 + 7, 320, 0.3, "adam", "bf16", "f32", "", "register"),
           (9, 2048 * 100 + 77, 2048, 0.3, "adam", "f32", "f32", "alg1", "bulk-copy wide"),  # what a packet's launch reads beside its slab
           (6, 320 * 5000 + 40, 320, 0.2, "adam", "bf16", "bf16", "bursty", "gather wide"),
           (16, 1024 * 40 + 21, 1024, 0.3, "sgd", "bf16", "bf16", "reliable", "bulk-copy")]


def _runs():
    out = []
    for q, (W, n, P, p, opt, g, r, mode, plan) in enumerate(BUCKETS):
        w = workload.Workload(f"b2b{q}", W, n, P, p, opt, 3e-4, g, r, 4, seed=31 + q)
        run = GpuRun(w, alg1=mode == "alg1", burst=(0.15, 0.4) if mode == "bursty" else None)
        if mode == "reliable":
            gen = torch.Generator(device="cuda").manual_seed(q)
            run.reliable = torch.randint(0, 1 << W, (2 * w.K,), generator=gen, device="cuda")
            L.lossy_set_reliable(run.ctx, run.reliable)
        assert L.lossy_describe_plan(run.ctx).startswith(plan)
        out.append((run, [workload.grad_slab(w, 1, i, 0, n, "cuda") for i in range(W)]))
    return out


def _steps(runs, sync, first, steps):
    for t in range(first, first + steps):
        for run, grads in runs:
            for g in grads:
                g.mul_(-0.75)                           # rewritten by the kernels right ahead of the step
            (run.step_fused if t % 3 else run.step_unfused)(t, grads)
            if sync:
                torch.cuda.synchronize()


def _same(a, b):
    for (x, _), (y, _) in zip(a, b):
        ox, oy = x.outputs(), y.outputs()
        for k in ox:
            assert_same(ox[k], oy[k], f"{x.w.name} {k}")
        for name in ("master", "m", "v", "ghat_prev", "burst_state"):
            if getattr(x, name) is None:
                continue
            assert_same(to_np(getattr(x, name)), to_np(getattr(y, name)), f"{x.w.name} {name}")
        for i in range(x.w.W):
            assert_same(to_np(x.replicas[i]), to_np(y.replicas[i]), f"{x.w.name} replica {i}")
        L.lossy_device_status(x.ctx)


def test_calls_without_a_pause_between_them():
    a, b = _runs(), _runs()
    torch.cuda.synchronize()
    _steps(a, False, 1, 9)
    _steps(b, True, 1, 9)
    _same(a, b)


def test_calls_in_a_graph_with_a_fork_and_a_join():
    a, b = _runs(), _runs()
    side, main = torch.cuda.Stream(), torch.cuda.Stream()
    torch.cuda.synchronize()
    for runs in (a, b):
        _steps(runs, True, 1, 3)                        # (every kernel has been launched once before the capture)
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=main):
        _steps(a[:2], False, 4, 3)
        side.wait_stream(main)
        with torch.cuda.stream(side):
            _steps(a[2:], False, 4, 3)                  # two branches of the graph, then a join
        _steps(a[:2], False, 7, 2)
        main.wait_stream(side)
        _steps(a[2:], False, 7, 2)
    for _ in range(2):                                  # (a replay makes the same calls again)
        g.replay()
        _steps(b, True, 4, 5)
    _same(a, b)
