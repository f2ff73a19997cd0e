"""Bursty loss on the gather pipeline: the mask warp holds a tile's link words a tile ahead. Several tiles per block, tiles that start inside
a packet, more than 32 workers (one packet per pass of draws), and a part-empty last tile, against the register kernel bit for
bit, link states included."""
import pytest
import torch

import paper_2507_07114_b200 as L
import workload
from parity_util import GpuRun, assert_rel, assert_same, to_np

CASES = [(12, 256 * 4700, 256, 0.1, "bf16", "bf16"), (3, 128 * 9000 + 40, 128, 0.3, "f32", "bf16"), (40, 512 * 1900, 512, 0.05, "bf16", "f32"),
         (9, 736 * 2300 + 5, 736, 0.2, "bf16", "bf16"), (33, 336 * 2800, 336, 0.1, "bf16", "bf16"), (17, 256 * 9, 256, 0.3, "bf16", "bf16")]


@pytest.mark.gpu
@pytest.mark.parametrize("W,n,P,p,g,r", CASES)
def test_link_words_a_tile_ahead(W, n, P, p, g, r):
    w = workload.Workload("burst_gather", W, n, P, p, "adam", 3e-4, g, r, 3, seed=n % 83)
    a, b = (GpuRun(w, flags=f, burst=(p / 3, 0.3)) for f in (L.LOSSY_GATHER_PATH, L.LOSSY_REGISTER_PATH))
    assert L.lossy_describe_plan(a.ctx).startswith("gather") and L.lossy_describe_plan(b.ctx).startswith("register")
    for t in (1, 2, 3):
        grads = [workload.grad_slab(w, t, i, 0, n, "cuda") for i in range(W)]
        a.step_fused(t, grads)
        b.step_fused(t, grads)
    oa, ob = a.outputs(), b.outputs()
    for k in ("ghat", "count", "recv_bits", "stale_bits"):
        assert_same(oa[k], ob[k], k)
    assert_rel(oa["sumsq"], ob["sumsq"], "drift sums", tol=1e-7)     # fp32 squares summed in other trees: 1e-8
    for name in ("master", "m", "v", "burst_state"):
        assert_same(to_np(getattr(a, name)), to_np(getattr(b, name)), name)
    for i in range(W):
        assert torch.equal(a.replicas[i], b.replicas[i]), f"replica {i}"
    L.lossy_device_status(a.ctx)
