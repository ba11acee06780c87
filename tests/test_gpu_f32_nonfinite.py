"""fp32 products of values that have no bf16 decomposition (infinities, NaN, magnitudes that round to infinity in
bf16): every epilogue, k cut over a cluster, CTA pairs and the short-contraction kernel behave as fp32 arithmetic,
and take a time of the same order."""
import pytest
import torch

from paper_1910_02120_b200 import api

pytestmark = pytest.mark.gpu


# classes = 64: one or a few tiles, k cut over clusters; 16385: pairs of CTAs; 33 inputs: CUDA cores or one step
@pytest.mark.parametrize("rows,n0,classes", [(9, 1025, 64), (100, 2000, 130), (300, 33, 40), (512, 300, 16385), (500, 129, 16384)])
def test_infinite_logits(rows, n0, classes):
    g = torch.Generator(device="cuda").manual_seed(classes)
    W = torch.rand(n0, classes, device="cuda", generator=g) + 0.25
    W *= torch.where(torch.rand(n0, classes, device="cuda", generator=g) < 0.3, 1.0, -1.0)
    X = torch.randn(rows, n0, device="cuda", generator=g)
    at = torch.arange(rows, device="cuda")
    hot = (at * 7 + 3) % n0
    X[at, hot] = float("inf")                             # logits -inf .. +inf by the sign of the weight
    y = (W[hot] > 0).int().argmax(1).int()                # the first +inf is the row's maximum
    assert bool((W[hot] > 0).any(1).all())
    ctx = api.Ist([n0, classes], 1, api.IST_FP32, 512)
    ctx.bind_weights([W], [torch.zeros(classes, device="cuda")])
    loss, hits = ctx.eval(X, y, rows)
    assert hits.item() == rows and loss.isnan().item()
    # one such row (and one of NaN) among ordinary ones: these do not see it
    clean = torch.randn(rows, n0, device="cuda", generator=g)
    z = (clean.double() @ W.double())
    best = z.argmax(1).int()
    mixed = clean.clone()
    mixed[rows // 2] = X[rows // 2]
    mixed[rows // 3] = float("nan")
    label = best.clone()
    label[rows // 2] = y[rows // 2]
    label[rows // 3] = classes - 1                        # no value is the largest: counted as wrong
    _, hits = ctx.eval(mixed, label, rows)
    ctx.sync_status()
    assert hits.item() == rows - 1


# (rows, inputs, hidden, classes): the second and third product have K = classes and K = rows
@pytest.mark.parametrize("B,n0,n1,n2", [(40, 30, 50, 20), (70, 90, 65, 300), (200, 129, 257, 1100), (128, 700, 70, 70),
                                        (640, 257, 4100, 1029), (161, 4100, 4099, 65)])
def test_values_that_round_to_infinity_in_bf16(B, n0, n1, n2):
    """Hidden neurons whose activation is 2e-38 and whose outgoing weights are 3.4e38: finite in every product,
    through the ReLU, mask, input-gradient and update epilogues."""
    g = torch.Generator(device="cuda").manual_seed(B)
    W1 = torch.randn(n0, n1, device="cuda", generator=g) / n0 ** 0.5
    W2 = torch.randn(n1, n2, device="cuda", generator=g) / n1 ** 0.5
    b1, b2 = torch.randn(n1, device="cuda", generator=g) * 0.1, torch.randn(n2, device="cuda", generator=g) * 0.1
    odd = torch.tensor([0, n1 // 2, n1 - 1], device="cuda")
    W1[:, odd], b1[odd] = 0.0, 2e-38
    W2[odd] = torch.where(torch.rand(3, n2, device="cuda", generator=g) < 0.5, 3.4e38, -3.4e38)
    X = 0.1 * torch.randn(B, n0, device="cuda", generator=g)
    y = torch.randint(n2, (B,), device="cuda", generator=g, dtype=torch.int32)
    lr = 1e-36
    a = (X.double() @ W1.double() + b1.double()).clamp_min(0)
    z = a @ W2.double() + b2.double()
    delta = torch.softmax(z, 1)
    delta[torch.arange(B), y.long()] -= 1
    delta /= B
    below = (delta @ W2.double().T) * (a > 0)
    assert below[:, odd].abs().max() > 1e35 and below.abs().max() < 3e38
    want_W1 = W1.double() - lr * (X.double().T @ below)
    want_dx = below @ W1.double().T                       # those neurons' weights are zero: they add nothing
    loss = torch.nn.functional.cross_entropy(z, y.long())

    W2_before = W2.clone()
    ctx = api.Ist([n0, n1, n2], 1, api.IST_FP32, B)
    ctx.bind_weights([W1, W2], [b1, b2])
    ctx.partition(3)
    dx = torch.empty(B, n0, device="cuda")
    got = ctx.local_steps(X, y, lr, 1, B, dx_out=dx)
    ctx.reassemble()
    ctx.sync_status()
    # ||difference|| as in test_gpu_f32_gemm.py, over two layers more; the input gradient's ReLU masks may flip where
    # a pre-activation is within rounding of zero
    tol = 2 ** -24 * (16 + n0 ** 0.5 + n1 ** 0.5 + max(B, n2) ** 0.5) * 2
    assert abs(got.item() - loss.item()) <= tol * max(1.0, abs(loss.item()))
    assert (W1[:, odd] - want_W1[:, odd]).norm() <= tol * want_W1[:, odd].norm()
    assert torch.equal(W2, W2_before)                     # lr * gradient is far below the last bit
    assert (dx - want_dx).norm() <= (tol + 1e-3) * want_dx.norm()


def _time(ctx, X, y, rows):
    best = 1e30
    for _ in range(3):
        t0, t1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        t0.record()
        ctx.eval(X, y, rows)
        t1.record()
        torch.cuda.synchronize()
        best = min(best, t0.elapsed_time(t1))
    return best


def test_overflow_costs_a_bounded_factor():
    """One hidden neuron at infinity makes every value behind it infinite.  The products are then formed on the CUDA
    cores, whose peak is a thirtieth of the bf16 tensor cores' and, six products for one, a fifth of theirs: 40 times
    leaves a factor of eight for the rest."""
    dims, rows = [256, 2048, 2048, 2048], 512
    g = torch.Generator(device="cuda").manual_seed(5)
    W = [torch.rand(a, b, device="cuda", generator=g) / a for a, b in zip(dims, dims[1:])]    # positive: no inf - inf
    b = [torch.zeros(n, device="cuda") for n in dims[1:]]
    X = torch.rand(rows, dims[0], device="cuda", generator=g)
    y = torch.zeros(rows, device="cuda", dtype=torch.int32)
    ctx = api.Ist(dims, 1, api.IST_FP32, rows)
    ctx.bind_weights(W, b)
    finite = _time(ctx, X, y, rows)
    b[0][1000] = float("inf")
    loss, hits = ctx.eval(X, y, rows)
    assert loss.isnan().item() and hits.item() == rows    # all logits are +inf: the first of them counts
    overflowed = _time(ctx, X, y, rows)
    ctx.sync_status()
    assert overflowed <= 40 * finite, (finite, overflowed)
