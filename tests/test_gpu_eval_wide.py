"""Evaluation over many classes: rows of every alignment, one to eight CTAs per row, ties, labels."""
import pytest
import torch

from paper_1910_02120_b200 import api

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("classes,rows", [(4095, 5), (4096, 5), (4099, 300), (8192, 2), (16386, 7), (70001, 3), (270003, 2),
                                          (600001, 1)])
def test_wide_rows(classes, rows):
    g = torch.Generator(device="cuda").manual_seed(classes)
    n0 = 32
    W = torch.randn(n0, classes, device="cuda", generator=g) / n0 ** 0.5
    b = torch.randn(classes, device="cuda", generator=g)
    lo, hi = classes // 3, classes - 1                # two classes tie for the maximum of every row
    W[:, hi] = W[:, lo]
    b[lo] = b[hi] = 40.0
    X = torch.randn(rows, n0, device="cuda", generator=g)
    y = torch.randint(classes, (rows,), device="cuda", generator=g, dtype=torch.int32)
    y[0] = lo
    y[-1] = hi if rows > 1 else lo
    want_hits = int((y == lo).sum())                  # the lower index counts
    want = torch.nn.functional.cross_entropy(X.double() @ W.double() + b.double(), y.long()).item()
    ctx = api.Ist([n0, classes], 1, api.IST_FP32, max(rows, 4))
    ctx.bind_weights([W], [b])
    loss, hits = ctx.eval(X, y, rows)
    ctx.sync_status()
    # the logits reach about 45: each is rounded at 2^-24 of that, once in the product and once with the
    # bias, and a row's loss is a difference of two such numbers
    assert abs(loss.item() - want) <= 4 * 2 ** -24 * 45 + 1e-6 * abs(want) and hits.item() == want_hits
    y[rows // 2] = classes
    ctx.eval(X, y, rows)
    with pytest.raises(api.IstError):
        ctx.sync_status()
