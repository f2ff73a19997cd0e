"""Calls of small buckets against calls that cannot be faster but by a fault of the launch: device times of captured calls, the better of
several replays, with a margin of several times what the replays differ by."""
import pytest
import torch

import paper_2507_07114_b200 as L
import workload
from parity_util import GpuRun

pytestmark = pytest.mark.gpu


def graph_times(*calls, repeats=30, replays=9):
    """us of each sequence of calls, captured `repeats` times, the sequences' graphs replayed in turn."""
    graphs = []
    for call in calls:
        stream, g = torch.cuda.Stream(), torch.cuda.CUDAGraph()
        stream.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(stream):
            call()
            torch.cuda.synchronize()
            with torch.cuda.graph(g, stream=stream):
                for _ in range(repeats):
                    call()
        graphs.append(g)
    best = [float("inf")] * len(calls)
    a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    for _ in range(replays):
        for k, g in enumerate(graphs):
            g.replay()
            a.record()
            g.replay()
            b.record()
            b.synchronize()
            best[k] = min(best[k], a.elapsed_time(b) / repeats * 1e3)
    return best


def make(W, n, P, p=0.1, g="bf16", r="bf16", optimizer="adam", flags=0):
    w = workload.Workload("times", W, n, P, p, optimizer, 3e-4, g, r, 2, seed=3)
    run = GpuRun(w, flags=flags)
    return run, [workload.grad_slab(w, 1, i, 0, n, "cuda") for i in range(W)]


@pytest.mark.parametrize("W,P", [(8, 512), (23, 2048), (53, 512)])
def test_a_step_of_few_chunks_is_no_slower_than_one_of_many(W, P):
    """The end of the drift norms sums every block's row for every replica. With one warp per block, as many as 2048 elements have
    chunks for, W = 53 took 27 us, with 37 k elements 14.5."""
    few, few_grads = make(W, 4 * P if P < 2048 else P, P, flags=L.LOSSY_REGISTER_PATH)
    many, many_grads = make(W, 36_864, P, flags=L.LOSSY_REGISTER_PATH)
    a, b = graph_times(lambda: few.step_fused(1, few_grads, outputs=False), lambda: many.step_fused(1, many_grads, outputs=False))
    assert a <= 1.15 * b, (a, b)


@pytest.mark.parametrize("W,n,P", [(6, 497_803, 6736), (2, 2_126_753, 8192)])
def test_packet_norms_right_behind_a_kernel(W, n, P):
    """A memset in front makes any kernel's launch an ordinary one. Blocks that begin while the pairwise drift still runs share the few SMs
    that it leaves first: with up to 592 of them 25 us for 12.5, memset included."""
    run, grads = make(W, n, P)
    d2, out, word = torch.zeros(W * W, dtype=torch.float64, device="cuda"), torch.empty(W * -(-n // P), device="cuda"), torch.zeros(1, device="cuda")

    def diagnostics(between):
        d2.zero_()
        L.drift_pairwise(run.ctx, run.replicas, d2)
        if between:
            word.zero_()
        L.lossy_packet_sqnorms(run.ctx, grads, out)

    a, b = graph_times(lambda: diagnostics(False), lambda: diagnostics(True))
    assert a <= 1.15 * b, (a, b)


@pytest.mark.parametrize("W,n,P", [(59, 321_136, 8192), (18, 157_952, 256), (31, 226_284, 4096)])
def test_closed_loop_gradients_right_behind_a_step(W, n, P):
    """The same for the gradients of the closed loop: with up to 444 blocks begun early 120 us for 95, 23 for 18 and 52 for 43."""
    run, grads = make(W, n, P, 0.01, "f32", "f32")
    noise, word = [g.clone() for g in grads], torch.zeros(1, device="cuda")
    curv, target = torch.full((n,), 0.7, device="cuda"), torch.zeros(n, device="cuda")

    def step(between):
        if between:
            word.zero_()
        L.lossy_closed_loop_grads(run.ctx, curv, target, noise, run.replicas, grads)
        run.step_fused(1, grads, outputs=False)

    a, b = graph_times(lambda: step(False), lambda: step(True))
    assert a <= 1.08 * b, (a, b)


@pytest.mark.parametrize("W,n,P", [(41, 374_272, 512), (63, 737_394, 256)])
def test_a_broadcast_right_behind_the_optimizer(W, n, P):
    """The same for the broadcast, of packets that no pipeline takes: with 183 blocks and 361 begun early the four phases took 73 us for 63
    and 203 for 157."""
    run, grads = make(W, n, P, 0.0 if P == 512 else 0.01, "bf16", "f32")
    word = torch.zeros(1, device="cuda")

    def step(between):
        L.lossy_aggregate(run.ctx, 1, grads, run.ghat)
        L.lossy_step(run.ctx, 1, run.ghat, None, run.master, run.m, run.v)
        if between:
            word.zero_()
        L.lossy_broadcast(run.ctx, 1, run.master, run.replicas)
        L.drift_norms(run.ctx, run.master, run.replicas, run.norms)

    a, b = graph_times(lambda: step(False), lambda: step(True))
    assert a <= 1.05 * b, (a, b)


@pytest.mark.parametrize("W,n,P", [(60, 74_933, 512)])
def test_a_bucket_that_ends_inside_eight_elements(W, n, P):
    """The lane that the end falls into loads and stores its few elements one by one, for every replica; the lanes behind it ran beside it
    before they skipped every access, and then behind it: broadcast of W = 60 9.0 us, 5.4 of the whole packets, 6.8 as it was."""
    (ragged, _), (whole, _) = make(W, n, P), make(W, -(-n // P) * P, P)
    a, b = graph_times(*(lambda x=x: L.lossy_broadcast(x.ctx, 1, x.master, x.replicas, x.stale) for x in (ragged, whole)))
    assert a <= 1.45 * b, (a, b)
