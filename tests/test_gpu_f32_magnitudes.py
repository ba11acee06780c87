"""fp32 products over fp32's whole range of exponents: scaling one operand by a power of two and the other by its
inverse changes no bit of the result, as in fp32 arithmetic; with operands whose low bf16 parts are subnormal numbers,
no more than the rounding of a single product."""
import pytest
import torch

from paper_1910_02120_b200 import api

pytestmark = pytest.mark.gpu


# one step on the CUDA cores, then the tensor cores: one tile, k cut over a cluster, several tiles, pairs of CTAs
@pytest.mark.parametrize("B,n0,n1", [(8, 16, 24), (31, 100, 65), (9, 1024, 64), (128, 520, 260), (512, 129, 16384), (640, 4100, 1029)])
@pytest.mark.parametrize("power", [-118, -111, -100, 100, 111, 118])
def test_power_of_two_scaling(B, n0, n1, power):
    g = torch.Generator(device="cuda").manual_seed(B)
    W = torch.randn(n0, n1, device="cuda", generator=g) / n0 ** 0.5
    b = torch.randn(n1, device="cuda", generator=g) * 0.1
    X = (torch.rand(B, n0, device="cuda", generator=g) + 0.25) * torch.randn(B, n0, device="cuda", generator=g).sign()
    W = torch.where(W.abs() < 2.0 ** -7, 2.0 ** -7, W)      # with the scaling all of them stay normal numbers
    y = torch.randint(n1, (B,), device="cuda", generator=g, dtype=torch.int32)
    out = []
    for p in (0, power):
        ctx = api.Ist([n0, n1], 1, api.IST_FP32, B)
        Wp = (W * 2.0 ** p).contiguous()
        ctx.bind_weights([Wp], [b.clone()])
        ctx.partition(1)
        dx = torch.empty(B, n0, device="cuda")
        loss = ctx.local_steps(X * 2.0 ** -p, y, 0.0, 1, B, dx_out=dx)
        ctx.reassemble()
        ctx.sync_status()
        out.append((loss, dx))
    (loss, dx), (loss_p, dx_p) = out
    want = dx.double() * 2.0 ** power
    assert torch.isfinite(loss).all()
    # results below 2^-126 are multiples of 2^-149, and a sum may lose one of them at each of the four places where it
    # is cut off: two rescalings and the last products of every 32 terms, and their addition
    tiny = 2 ** -149 * 4 * (-(-n1 // 32)) * want.numel() ** 0.5
    if abs(power) == 118:                                   # W or X down to 2^-125: their low bf16 parts are subnormal numbers
        assert abs(loss_p.item() - loss.item()) <= 2 ** -23 * loss.item()
        assert (dx_p.double() - want).norm() <= 2 ** -25 * want.norm() + tiny
    elif power > 0:
        assert torch.equal(loss, loss_p) and torch.equal(dx_p.double(), want)
    else:
        # deltas of improbable classes are small already; scaled down as well, results leave the normal range
        assert torch.equal(loss, loss_p)
        assert (dx_p.double() - want).norm() <= 2 ** -25 * want.norm() + tiny
