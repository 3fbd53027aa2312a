"""The tensor core adds products of 8-bit integers held as FP16 without rounding
up to 2^24 in its FP32 accumulators, which the digit-plane transforms rest on:
1024 products of one sign up to the largest sum, with odd remainders, and of
mixed signs."""
import pytest
import torch

from tests.gpu_util import ctx

pytestmark = pytest.mark.gpu


def _operand(rows, kind, g):
    if kind == "largest":
        return torch.full((1, rows, 1024), -128)
    if kind == "odd":
        return torch.full((1, rows, 1024), 127)
    lo, hi = (101, 128) if kind == "one sign" else (-128, 128)
    return torch.randint(lo, hi, (1, rows, 1024), generator=g)


@pytest.mark.parametrize("kind", ["largest", "odd", "one sign", "mixed"])
@pytest.mark.parametrize("N", [16, 128])
def test_integer_sums_up_to_the_full_range(kind, N):
    c = ctx()
    g = torch.Generator().manual_seed(N)
    a, b = _operand(128, kind, g), _operand(N, kind, g)
    want = (a.double() @ b.double().transpose(1, 2)).long()
    assert int(want.abs().max()) <= 1 << 24
    ah, bh = a.half().cuda(), b.half().cuda()
    d = c.gemm_f16x3(ah, torch.zeros_like(ah), bh, torch.zeros_like(bh))
    c.sync()
    assert torch.equal(d.cpu().double().long(), want)
