"""Packet norms, pairwise drift and the closed loop's gradients right behind calls that write what they read, and in front of calls that
write what they have read: without a pause and in a graph they give what calls with a synchronisation after each give. On both sides
of the lines up to which they begin while the kernel ahead still runs, and of those between their builds."""
import pytest
import torch

import paper_2507_07114_b200 as L
import workload
from parity_util import GpuRun, assert_rel, assert_same, to_np

pytestmark = pytest.mark.gpu

# W, n, P, types. Packet norms begin early under 16 blocks of eight pieces (packets up to 256 elements: of 32), the closed loop's gradients up to
# 64 blocks of 2048 elements, with two or three workers up to 444; the pairwise drift has a build for up to eight replicas of
# 303 104 elements and one for more (its lines are for 148 SMs).
BUCKETS = [(3, 20_003, 2048, "bf16", "bf16"),       # few replicas, norms and gradients early
           (3, 900_000, 8192, "bf16", "f32"),       # 440 blocks of gradients, early
           (8, 131_072, 1024, "f32", "bf16"),       # 64 blocks, 128 of the norms
           (8, 133_120, 256, "bf16", "bf16"),       # 65 blocks
           (12, 60_008, 8192, "bf16", "bf16"),      # the small set build; 12 blocks of norms
           (12, 400_000, 128, "f32", "f32"),        # the large one
           (40, 30_001, 512, "bf16", "f32"),        # sets of 64 bits, 320 blocks of norms
           (2, 8 * 1024 * 7, 1024, "f32", "f32")]   # 14 blocks of norms


def _runs():
    out = []
    for q, (W, n, P, g, r) in enumerate(BUCKETS):
        w = workload.Workload(f"diag{q}", W, n, P, 0.2, "adam", 3e-4, g, r, 4, seed=51 + q)
        run = GpuRun(w)
        run.noise = [workload.grad_slab(w, 1, i, 0, n, "cuda") for i in range(W)]
        run.grads = [torch.zeros_like(x) for x in run.noise]
        run.curv, run.target = torch.linspace(0.5, 1.5, n, device="cuda"), torch.linspace(-0.02, 0.02, n, device="cuda")
        run.d2 = torch.zeros(W * W, dtype=torch.float64, device="cuda")
        run.sq, run.sq_before = (torch.zeros(W * w.K, device="cuda") for _ in range(2))
        out.append(run)
    return out


def _steps(runs, sync, first, steps):
    for t in range(first, first + steps):
        for run in runs:
            calls = [lambda: L.lossy_packet_sqnorms(run.ctx, run.grads, run.sq_before),                              # behind the drift of the step before,
                     lambda: L.lossy_closed_loop_grads(run.ctx, run.curv, run.target, run.noise, run.replicas, run.grads),   # in front of what rewrites it,
                     lambda: L.lossy_packet_sqnorms(run.ctx, run.grads, run.sq),                                     # behind what wrote it
                     lambda: run.step_fused(t, run.grads, outputs=False),
                     lambda: L.drift_pairwise(run.ctx, run.replicas, run.d2)]                                        # behind the step that wrote the replicas
            for call in calls:
                call()
                if sync:
                    torch.cuda.synchronize()


def _same(a, b):
    torch.cuda.synchronize()
    for x, y in zip(a, b):
        for name in ("master", "m", "v", "sq", "sq_before"):
            assert_same(to_np(getattr(x, name)), to_np(getattr(y, name)), f"{x.w.name} {name}")
        for i in range(x.w.W):
            assert_same(to_np(x.replicas[i]), to_np(y.replicas[i]), f"{x.w.name} replica {i}")
            assert_same(to_np(x.grads[i]), to_np(y.grads[i]), f"{x.w.name} gradients {i}")
        assert_rel(to_np(x.d2), to_np(y.d2), f"{x.w.name} pairwise drift", tol=1e-12)        # fp64 atomics in any order
        L.lossy_device_status(x.ctx)


def test_diagnostics_without_a_pause():
    a, b = _runs(), _runs()
    torch.cuda.synchronize()
    _steps(a, False, 1, 8)
    _steps(b, True, 1, 8)
    _same(a, b)


def test_diagnostics_in_a_graph():
    a, b = _runs(), _runs()
    torch.cuda.synchronize()
    for runs in (a, b):
        _steps(runs, True, 1, 2)
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=torch.cuda.Stream()):
        _steps(a, False, 3, 4)
    for _ in range(2):
        g.replay()
        _steps(b, True, 3, 4)
    _same(a, b)
