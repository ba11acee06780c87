"""The loss's exponentials are added in one fixed order, whichever kernel a class count goes to: the sum over
a row of up to 1024 classes is that of a block of 32 (up to 64 classes) or 128 threads with strided
columns.  The order is part of the results: a last bit of the sum moves roundings of the deltas to bf16, and a
few steps of a bf16 network make 1e-4 of it."""
import pytest
import torch

from paper_1910_02120_b200 import api

pytestmark = pytest.mark.gpu


def _sum_in_order(e, threads):
    """Strided partial sums of `threads` threads, a butterfly within each warp, then one over the warps."""
    n = -(-e.numel() // threads) * threads
    cols = torch.zeros(n, device=e.device).index_copy_(0, torch.arange(e.numel(), device=e.device), e).view(-1, threads)
    part = cols[0].clone()
    for row in cols[1:]:
        part = part + row
    lanes = part.view(-1, 32)
    for o in (16, 8, 4, 2, 1):
        lanes = lanes + lanes[:, torch.arange(32, device=e.device) ^ o]
    warps = torch.zeros(32, device=e.device)
    warps[:lanes.shape[0]] = lanes[:, 0]
    for o in (16, 8, 4, 2, 1):
        warps = warps + warps[torch.arange(32, device=e.device) ^ o]
    return warps[0]


@pytest.mark.parametrize("classes", [2, 33, 64, 65, 96, 100, 128, 129, 300, 512, 513, 1000, 1024])
def test_sum_of_exponentials_has_a_fixed_order(classes):
    # no hidden layer and a row of zeros: the logits are the bias, bit for bit; one row: delta is p - [n == y]
    g = torch.Generator(device="cuda").manual_seed(classes)
    W, b = torch.zeros(8, classes, device="cuda"), torch.zeros(classes, device="cuda")
    ctx = api.Ist([8, classes], 1, api.IST_FP32, 1)
    ctx.bind_weights([W], [b])
    X, y = torch.zeros(1, 8, device="cuda"), torch.zeros(1, dtype=torch.int32, device="cuda")
    lr = 2.0 ** 20                                      # a power of two: lr * delta is exact
    for i in range(8):
        z = 2.0 * torch.randn(classes, device="cuda", generator=g)
        b.copy_(z)
        ctx.partition(i)
        ctx.local_steps(X, y, lr, 1, 1)
        ctx.reassemble()
        ctx.sync_status()
        e = torch.exp(z - z.max())
        p = e * (1.0 / _sum_in_order(e, 32 if classes <= 64 else 128))
        # the update is one multiply-add, rounded once; column 0 holds the label
        want = (z.double() - lr * p.double()).float()
        assert torch.equal(b[1:], want[1:]), i
