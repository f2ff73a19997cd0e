"""Four workers at little loss: where whole packets leave the step kernel, and that nothing else leaves it with them (148 SMs, tiles of
2048 elements)."""
import pytest
import torch

import paper_2507_07114_b200 as L

pytestmark = pytest.mark.gpu
SM_TILE = 148 * 2048


@pytest.mark.parametrize("P,inside,outside,rest,plan", [(400, 6.7, 6.8, 10.9, "gather wide"), (168, 6.7, 6.8, 10.9, "gather twin"), (4944, 5.7, 5.8, 6.9, "bulk-copy twin")])
def test_lines_of_four_workers(P, inside, outside, rest, plan):
    def kernel(tiles, W=4, p=0.05, g="bf16", r="bf16", optimizer="adam", flags=0, extra=0):
        dtype = {"bf16": torch.bfloat16, "f32": torch.float32}
        ctx = L.lossy_init(W=W, n=int(tiles * SM_TILE) // P * P + extra, packet_elems=P, p_grad=p, p_param=p, seed=1, grad_dtype=dtype[g],
                           replica_dtype=dtype[r], optimizer=optimizer, lr=1e-3, flags=flags)
        try:
            assert L.lossy_describe_plan(ctx).startswith(L.lossy_describe_plan(ctx, with_drift=False))    # with drift norms and without
            return L.lossy_describe_plan(ctx)
        finally:
            L.lossy_destroy(ctx)

    assert kernel(inside) == "register kernel"
    assert kernel(outside).startswith(plan) and kernel(outside, p=0.0, g="f32").startswith(plan) and kernel(rest).startswith(plan)
    for tiles in (outside, rest):
        for other in ({"p": 0.1}, {"W": 3}, {"W": 2}, {"r": "f32"}, {"optimizer": "sgd"}, {"flags": L.LOSSY_REPLICA_SKIP_OWNER}, {"extra": 8}):
            assert kernel(tiles, **other) == "register kernel", other
