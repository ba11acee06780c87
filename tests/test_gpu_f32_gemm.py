"""fp32 products at the edges of their tiles, against 64-bit arithmetic.

A network without hidden layers has no ReLU whose mask could flip, so one local step checks the three
kinds of product by themselves: z = X W + b through the loss, d(loss)/dX = delta W^T, and W - lr X^T delta."""
import pytest
import torch

from paper_1910_02120_b200 import api, synth
from tests import helpers as H

pytestmark = pytest.mark.gpu


# 16 / 17 k values: the line to the short-contraction kernel; 64 / 65: its end; 31..33 and 127..129: edges
# of a step and of a tile; odd widths: rows without 16-byte alignment; few tiles and a deep sum: k cut
# over a cluster; (640, 2048, 4100) and (511, ...): pairs of CTAs in the forward product and the update, (640, 4100,
# 1029) in the input gradient as well; the last four: pairs whose update takes 5 to 9 steps through four operand slots.
SIZES = [(1, 1, 1), (5, 16, 3), (24, 33, 17), (31, 65, 64), (33, 64, 16), (128, 128, 128), (129, 127, 65), (64, 5000, 130),
         (200, 1001, 777), (40, 64, 512), (40, 64, 513), (9, 64, 1024), (9, 64, 1025), (640, 2048, 4100), (511, 1029, 8209),
         (640, 4100, 1029),
         (129, 4100, 4099), (161, 4099, 4100), (225, 4100, 4100), (260, 4099, 4099)]


@pytest.mark.parametrize("B,n0,n1", SIZES)
def test_products_of_one_step(B, n0, n1):
    g = torch.Generator(device="cuda").manual_seed(B * 7 + n0)
    W = torch.randn(n0, n1, device="cuda", generator=g) / n0 ** 0.5
    b = torch.randn(n1, device="cuda", generator=g) * 0.1
    X = torch.randn(B, n0, device="cuda", generator=g)
    y = torch.randint(n1, (B,), device="cuda", generator=g, dtype=torch.int32)
    lr = 0.5 * B                                    # an update of the weights' own size
    z = X.double() @ W.double() + b.double()
    delta = torch.softmax(z, 1)
    delta[torch.arange(B), y.long()] -= 1
    delta /= B
    loss = torch.nn.functional.cross_entropy(z, y.long())
    grad = X.double().T @ delta
    want_W, want_dx = W.double() - lr * grad, delta @ W.double().T

    ctx = api.Ist([n0, n1], 1, api.IST_FP32, B)
    ctx.bind_weights([W], [b])
    ctx.partition(3)
    dx = torch.empty(B, n0, device="cuda")
    got = ctx.local_steps(X, y, lr, 1, B, dx_out=dx)
    ctx.reassemble()
    ctx.sync_status()
    # A 32-bit sum of K terms is off by at most about sqrt(K) 2^-24 of its size with random roundings; the
    # logits' error (K = n0 <= 5000: 4e-6 at worst) goes through the softmax into everything else.
    tol = 2 ** -24 * (8 + n0 ** 0.5 + max(B, n1) ** 0.5)
    assert abs(got.item() - loss.item()) <= tol * max(1.0, abs(loss.item()))
    assert (dx - want_dx).norm() <= tol * want_dx.norm()
    # the weight itself is rounded once more
    assert (W - want_W).norm() <= tol * lr * grad.norm() + 2 ** -24 * want_W.norm()


def test_values_without_a_bf16_decomposition():
    """Magnitudes that round to infinity in bf16, and infinities, behave as in fp32 arithmetic."""
    n0, n1 = 128, 40
    W = torch.full((n0, n1), 0.25, device="cuda")
    W[0] = torch.linspace(-1e-38, 1e-38, n1, device="cuda")
    W[1] = torch.linspace(-1.0, 1.0, n1, device="cuda")     # no zero among them
    b = torch.zeros(n1, device="cuda")
    X = torch.zeros(3, n0, device="cuda")
    X[0, 0] = 3.4e38                                        # finite products of a huge and a tiny number
    X[1, 1] = float("inf")                                  # logits -inf .. +inf; the other rows must not see them
    X[2, 2] = 1.0
    y = torch.tensor([n1 - 1, 20, 0], device="cuda", dtype=torch.int32)
    ctx = api.Ist([n0, n1], 1, api.IST_FP32, 4)
    ctx.bind_weights([W], [b])
    z = X[0].double() @ W.double()
    loss, hits = ctx.eval(X[:1].contiguous(), y[:1].contiguous(), 1)
    assert abs(loss.item() - torch.nn.functional.cross_entropy(z, y[0].long()).item()) <= 1e-5 and hits.item() == 1
    _, hits = ctx.eval(X[1:2].contiguous(), y[1:2].contiguous(), 1)
    assert hits.item() == 1                                 # the first +inf among the logits is class 20
    loss, _ = ctx.eval(X[2:].contiguous(), y[2:].contiguous(), 1)
    assert abs(loss.item() - torch.log(torch.tensor(float(n1))).item()) <= 1e-5
    ctx.sync_status()


# 256 blocks of bias work ride on the update launch, 368 go out as a launch of their own (the line is 296)
@pytest.mark.parametrize("classes", [700, 1100])
@pytest.mark.parametrize("B", [20, 70])
def test_bias_updates_beside_and_before_the_weight_updates(classes, B):
    w = synth.Workload("bias", (20, 3200, classes), S=16, B=B, K=2, rounds=1, precision="fp32", x_dist="normal", lr=0.5, seed=B)
    W, b, data = H.make_problem(w)
    o, _, oloss = H.oracle_round(w, W, b, data, 5)
    _, gW, gb, _, gloss = H.gpu_round(w, W, b, data, 5)
    H.assert_close(gloss, oloss, 1e-4, "losses")
    for l in range(len(W)):
        H.assert_close(gW[l], o.W[l], 1e-4, f"W_{l + 1}")
        H.assert_close(gb[l] - b[l], o.b[l] - b[l], 1e-3, f"update of b_{l + 1}")


@pytest.mark.parametrize("B,n0,n1", [(64, 512, 64), (1024, 512, 64), (16384, 512, 64), (1024, 4096, 4096)])
def test_mean_signed_error(B, n0, n1):
    """Accumulation that cuts off instead of rounding has a sign.  Logits far apart make every row's delta +-1/B in two
    columns, so the update there is the mean of X's rows and all products are exact: what is seen is the summing.  Sums
    of positive terms, the worst case, stay within the rounding of one number on average; their spread is that of B / 32
    additions, each off by a uniform share of 2^-24 of a sum that grows to its end, beside a few roundings."""
    g = torch.Generator(device="cuda").manual_seed(B)
    X = torch.rand(B, n0, device="cuda", generator=g) + 0.5
    W, b = torch.zeros(n0, n1, device="cuda"), torch.zeros(n1, device="cuda")
    b[0] = 300.0
    ctx = api.Ist([n0, n1], 1, api.IST_FP32, B)
    ctx.bind_weights([W], [b])
    ctx.partition(1)
    ctx.local_steps(X, torch.ones(B, device="cuda", dtype=torch.int32), -1.0, 1, B)
    ctx.reassemble()
    ctx.sync_status()
    want = X.double().mean(0)
    for column in (W[:, 0], -W[:, 1]):
        err = (column.double() - want) / want
        assert err.mean().abs() <= 2 ** -24 and err.square().mean().sqrt() <= 2 ** -24 * (4 + (B / 32) ** 0.5 / 4)
