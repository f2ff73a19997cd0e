"""Precision of a step's drift sums on the register kernel, which takes small buckets from pipelines that widen to fp64 after 128
squares: it must not be coarser than they are."""
import pytest
import torch

import paper_2507_07114_b200 as L
import workload
from parity_util import GpuRun

pytestmark = pytest.mark.gpu
SM_TILE = 148 * 2048
# W, n, P, p, replicas, flags: one to several stale copies per packet, short last packets, packets that leave lanes idle
CASES = [(8, 2 * SM_TILE - 512, 512, 0.2, "bf16", 0), (4, 2 * SM_TILE - 256 + 40, 256, 0.3, "bf16", 0), (16, SM_TILE + 1003, 4480, 0.3, "bf16", 0),
         (33, 2 * SM_TILE + 77, 2048, 0.1, "bf16", 0), (9, SM_TILE - 256, 256, 0.2, "f32", 0), (8, 520 * 900, 520, 0.3, "bf16", L.LOSSY_REGISTER_PATH),
         (64, SM_TILE, 1024, 0.3, "bf16", L.LOSSY_REGISTER_PATH)]


@pytest.mark.parametrize("W,n,P,p,r,flags", CASES)
def test_drift_sums_are_fp64_from_the_lane_on(W, n, P, p, r, flags):
    """Copies N(0, 3e-4) apart, as a training run has them. Eight bf16 squares added in fp32 and everything else in fp64 come out
    3.4e-10 low (the same order in NumPy; eight fp32 ones 3e-10 at this size), a warp's tree of 256 squares in fp32 8.8e-9,
    of 128 squares 6.0e-9."""
    w = workload.Workload("precision", W, n, P, p, "sgd", 0.0, "bf16", r, 1, seed=n % 89)
    gpu = GpuRun(w, flags=flags)
    assert L.lossy_describe_plan(gpu.ctx).startswith("register")
    torch.manual_seed(W)
    for rep in gpu.replicas:
        rep.copy_(gpu.master + 3e-4 * torch.randn(n, device="cuda"))
    grads = [torch.zeros(n, device="cuda", dtype=torch.bfloat16) for _ in range(W)]
    gpu.step_fused(1, grads)
    wire = gpu.master.to(gpu.replicas[0].dtype).double()
    want = torch.stack([((rep.double() - wire) ** 2).sum() for rep in gpu.replicas])
    assert abs(float(gpu.sumsq.sum() / want.sum()) - 1) <= 1.5e-9
    assert torch.all((gpu.sumsq - want).abs() <= 6e-7 * want)   # each: ten roundings by 2^-24 at most
