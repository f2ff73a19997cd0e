"""The register kernel divides a sum by the received count as a product with the reciprocal, corrected once by its exact
remainder: for every count up to 64 that is the IEEE quotient of every mantissa, and sums too small for it (or infinite, or
NaN) take the division. Here for all 2^23 mantissas, and around the line between the two."""
import pytest
import torch

import paper_2507_07114_b200 as L

pytestmark = pytest.mark.gpu
N = 1 << 23


def _quotients(W, sums, zeros):
    """sums / W through lossy_aggregate: one worker sends the sums, the others zeros, nothing is lost."""
    n = sums.numel()
    ctx = L.lossy_init(W=W, n=n, packet_elems=256, p_grad=0.0, p_param=0.0, seed=1, grad_dtype=torch.float32,
                       replica_dtype=torch.float32, optimizer="sgd", lr=0.1, flags=L.LOSSY_REGISTER_PATH)
    ghat = torch.empty_like(sums)
    L.lossy_aggregate(ctx, 1, [sums] + [zeros[:n]] * (W - 1), ghat)
    torch.cuda.synchronize()
    L.lossy_destroy(ctx)
    return ghat


def _ieee(sums, W):
    # the fp64 quotient of an fp32 value and a count below 2^7 rounds to fp32 as the exact one does (53 >= 2 * 24 + 2 bits)
    return (sums.double() / W).float()


def test_every_mantissa_of_every_count():
    zeros = torch.zeros(N, device="cuda")
    sums = (torch.arange(N, device="cuda", dtype=torch.int32) | 0x3F800000).view(torch.float32)
    for W in range(2, 65):
        assert torch.equal(_quotients(W, sums, zeros), _ieee(sums, W)), f"count {W}"


@pytest.mark.parametrize("W", [3, 7, 13, 48, 63, 64])
def test_sums_around_the_line_to_the_division(W):
    zeros = torch.zeros(N, device="cuda")
    gen = torch.Generator(device="cuda").manual_seed(W)
    rows = []
    for e in [0, 1, 2, 5, 6, 7, 8, 9, 10, 127, 200, 253, 254, 255]:     # biased exponents: subnormal, the line at 8, infinity and NaN
        mant = torch.randint(0, 1 << 23, (4096,), generator=gen, device="cuda", dtype=torch.int32)
        mant[:2] = torch.tensor([0, (1 << 23) - 1], device="cuda", dtype=torch.int32)
        rows.append((mant | (e << 23)).view(torch.float32))
    sums = torch.cat(rows)
    sums = torch.cat([sums, -sums, torch.zeros(512, device="cuda")])
    sums = torch.cat([sums, sums[torch.randperm(sums.numel(), generator=gen, device="cuda")]])   # and mixed within a lane
    got, want = _quotients(W, sums, zeros), _ieee(sums, W)
    want = torch.where(sums == 0, torch.zeros_like(want), want)          # (a sum that starts at +0 is never -0)
    assert torch.equal(torch.isnan(got), torch.isnan(want))
    ok = ~torch.isnan(want)
    assert torch.equal(got[ok].view(torch.int32), want[ok].view(torch.int32))
