"""The fused step's register kernel in each of its builds, at the edges of its chunks, rounds and tasks, against the pipelines bit for
bit (whose parity with the oracle has tests of its own)."""
import pytest
import torch

import paper_2507_07114_b200 as L
import workload
from parity_util import GpuRun, assert_rel, assert_same, run_parity, to_np

SMS = 148
REG, ELIDE, PACKED, GATHER = L.LOSSY_REGISTER_PATH, L.LOSSY_REPLICA_SKIP_OWNER, L.LOSSY_PACKED_BULK, L.LOSSY_GATHER_PATH
# W, n, P, p, gradients, replicas, optimizer, further flags, and the build, a block's warps and their rounds (148 SMs). A bucket that ends
# inside a lane has a task more than chunks.
CASES = [
    (4, SMS * 32 * 128, 1024, 0.1, "f32", "f32", "sgd", 0, "few warps=32 rounds=1"),           # up to four workers: one full round,
    (2, SMS * 32 * 128 + 3, 1024, 0.3, "bf16", "bf16", "adam", 0, "few warps=17 rounds=2"),    # and three elements more, which are a second one
    (3, 136 * 900 + 1, 136, 0.2, "bf16", "f32", "adam", ELIDE, "few warps=13 rounds=1"),       # chunks that the packet does not fill
    (9, 2048 * 40 + 1, 2048, 0.3, "bf16", "bf16", "adam", 0, "pairs warps=9 rounds=1"),        # two elements per lane: a lone last one
    (64, 1024 * 60 + 1023, 1024, 0.3, "f32", "f32", "sgd", 0, "pairs warps=8 rounds=1"),       # 64 workers, nineteen stale copies: batches of four
    (33, 512 * 100, 512, 0.2, "bf16", "bf16", "adam", ELIDE, "pairs warps=8 rounds=1"),        # fewer chunks than the norms have warps for
    (17, SMS * 32 * 64, 256, 0.1, "bf16", "f32", "adam", 0, "pairs warps=32 rounds=1"),        # the last bucket of one round
    (8, SMS * 24 * 128, 256, 0.05, "bf16", "bf16", "adam", 0, "quads warps=24 rounds=1"),      # four per lane: one full round,
    (8, SMS * 24 * 128 + 2, 256, 0.05, "f32", "bf16", "adam", 0, "quads warps=13 rounds=2"),   # and two elements more
    (16, 736 * 500 + 5, 736, 0.1, "f32", "f32", "sgd", ELIDE, "quads warps=11 rounds=2"),
    (12, 1024 * 400 + 1022, 1024, 0.3, "bf16", "bf16", "adam", 0, "stale warps=22 rounds=1"),  # eight stale copies at a time
    (20, 128 * 9000 + 7, 128, 0.3, "bf16", "bf16", "adam", 0, "octs warps=16 rounds=4"),       # eight per lane, half of the lanes, seven behind the last
    (40, 1024 * 1000, 1024, 0.3, "f32", "bf16", "sgd", ELIDE, "octs warps=10 rounds=3"),
]


@pytest.mark.gpu
@pytest.mark.parametrize("case", CASES, ids=["W%d-n%d-P%d-p%g-%s-%s-%s-%d" % c[:8] for c in CASES])
def test_builds_against_the_pipelines(case):
    W, n, P, p, g, r, opt, flags, build = case
    w = workload.Workload("step", W, n, P, p, opt, 3e-4, g, r, 2, seed=n % 89)
    a, b = GpuRun(w, flags=flags | REG), GpuRun(w, flags=flags | (PACKED if P >= 1024 else GATHER))
    assert L.lossy_describe_plan(a.ctx, build=True) == "register kernel " + build
    assert L.lossy_describe_plan(a.ctx) == "register kernel" and not L.lossy_describe_plan(b.ctx, build=True).startswith("register")
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


@pytest.mark.gpu
@pytest.mark.parametrize("W,n,P", [(1, 3, 8), (3, 1024 + 5, 1024), (7, 8 * 33 + 7, 8), (64, 4096 + 2, 4096), (16, 200 * 9 + 199, 200)])
def test_tiny_buckets_against_the_oracle(W, n, P):
    run_parity(workload.Workload("step_tiny", W, n, P, 0.3, "adam", 3e-4, "bf16", "f32", 3, seed=5), 3, flags=REG)

