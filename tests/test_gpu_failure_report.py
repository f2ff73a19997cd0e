"""The library's failure report, exercised without a failure: a bounded wait that runs out sets the context's
status word; nothing faults, traps or hangs, and the context works again after a reset."""
import ctypes

import pytest
import torch

import paper_2507_07114_b200 as L
import workload
from parity_util import GpuRun, run_parity

pytestmark = pytest.mark.gpu


def test_a_wait_that_runs_out_is_reported_and_the_context_recovers():
    w = workload.scaled(workload.baseline_workloads()["cfg2_w8_layer_adam"], 2048 * 40 + 16)
    gpu, orc = run_parity(w, 2)                         # a healthy context: status is clean
    L.lossy_device_status(gpu.ctx)
    before = L.lossy_kernel_launches(gpu.ctx)
    L.lossy_selftest_wait_expiry(gpu.ctx, 1024)         # one small block waits on a barrier nothing completes
    with pytest.raises(L.LossyError) as ei:
        L.lossy_device_status(gpu.ctx)
    assert ei.value.code == L.LOSSY_EDEVICE
    assert L.lossy_kernel_launches(gpu.ctx) == before + 1
    with pytest.raises(L.LossyError) as ei:             # sticky until it is cleared
        L.lossy_device_status(gpu.ctx)
    assert ei.value.code == L.LOSSY_EDEVICE
    L.lossy_reset_status(gpu.ctx)
    L.lossy_device_status(gpu.ctx)
    # the CUDA context is intact and the same lossy context still computes what the oracle computes
    from parity_util import compare_outputs, compare_state, to_np
    for t in (3, 4):
        gs = [workload.grad_slab(w, t, i, 0, w.n) for i in range(w.W)]
        gpu.step_fused(t, [g.cuda() for g in gs])
        ref = orc.step(t, [to_np(g) for g in gs])
        compare_outputs(gpu.outputs(), ref, f"after reset, step {t}")
        compare_state(gpu, orc, f"after reset, step {t}")
    L.lossy_device_status(gpu.ctx)


@pytest.mark.parametrize("W,n,P,plan", [(4, 1024 * 40, 1024, "bulk-copy"), (4, 64 * 10, 64, "register")])
def test_a_failed_launch_is_reported_once(W, n, P, plan):
    """The runtime refuses a launch into a capture that has been invalidated (here by a synchronisation). The call says so,
    and a launch behind it that goes well is not reported as failed."""
    w = workload.Workload("refused", W, n, P, 0.1, "sgd", 1e-2, "f32", "f32", 2, seed=5)
    gpu, want = GpuRun(w), GpuRun(w)
    assert L.lossy_describe_plan(gpu.ctx).startswith(plan)
    grads = [workload.grad_slab(w, 1, i, 0, n, "cuda") for i in range(W)]
    ids = torch.arange(256, device="cuda", dtype=torch.int32)
    packet, out = torch.arange(256, device="cuda", dtype=torch.int64), torch.zeros(256, dtype=torch.uint8, device="cuda")
    stream, rt = torch.cuda.Stream(), ctypes.CDLL("libcudart.so.12")
    handle, graph = ctypes.c_void_p(stream.cuda_stream), ctypes.c_void_p()
    step = L.lossy_fused_step_prepared(gpu.ctx, grads, gpu.master, None, None, gpu.replicas, norms=gpu.norms, stream=stream)
    step(1)                                                 # (what a kernel's first launch sets up is not captured)
    want.step_fused(1, grads, outputs=False)
    torch.cuda.synchronize()
    launches = L.lossy_kernel_launches(gpu.ctx)
    assert rt.cudaStreamBeginCapture(handle, 1) == 0
    assert rt.cudaStreamSynchronize(handle) != 0
    with pytest.raises(L.LossyError) as ei:
        step(2)
    rt.cudaStreamEndCapture(handle, ctypes.byref(graph))
    rt.cudaGetLastError()                                   # (torch's runtime: this test's own two errors)
    assert ei.value.code == L.LOSSY_ECUDA and L.lossy_kernel_launches(gpu.ctx) == launches
    L.lossy_mask_grid(gpu.ctx, 1, ids, ids, packet, out)
    step(2)
    want.step_fused(2, grads, outputs=False)
    torch.cuda.synchronize()
    assert torch.equal(gpu.master, want.master) and torch.equal(gpu.norms, want.norms)
    L.lossy_device_status(gpu.ctx)


def test_selftest_arguments_are_checked():
    ctx = L.lossy_init(W=2, n=64, packet_elems=64, p_grad=0.1, p_param=0.1, seed=0, grad_dtype=torch.float32,
                       replica_dtype=torch.float32, optimizer="sgd", lr=0.1)
    for bad in (0, (1 << 20) + 1):
        with pytest.raises(L.LossyError) as ei:
            L.lossy_selftest_wait_expiry(ctx, bad)
        assert ei.value.code == L.LOSSY_EINVAL
    L.lossy_device_status(ctx)
    assert L.lossy_kernel_launches(ctx) == 0
    L.lossy_destroy(ctx)


def test_step_zero_is_rejected_by_every_entry_point_that_hashes_the_step():
    n = 1024 * 4
    ctx = L.lossy_init(W=2, n=n, packet_elems=1024, p_grad=0.1, p_param=0.1, seed=0, grad_dtype=torch.float32,
                       replica_dtype=torch.float32, optimizer="sgd", lr=0.1)
    z = [torch.zeros(n, device="cuda") for _ in range(2)]
    count = torch.zeros(4, dtype=torch.uint8, device="cuda")
    for call in (lambda: L.lossy_aggregate(ctx, 0, z, z[0], count),
                 lambda: L.lossy_aggregate_alg1(ctx, 0, z, z[1], z[0], count),
                 lambda: L.lossy_step(ctx, 0, z[0], count, z[1]),
                 lambda: L.lossy_broadcast(ctx, 0, z[0], z),
                 lambda: L.lossy_fused_step(ctx, 0, z, z[0], None, None, z)):
        with pytest.raises(L.LossyError) as ei:
            call()
        assert ei.value.code == L.LOSSY_EINVAL
    assert L.lossy_kernel_launches(ctx) == 0
    L.lossy_destroy(ctx)
