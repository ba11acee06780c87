"""Masters kept as bf16 operand and low half: every number is kept bit for bit, gathered or computed, the operand
is the master rounded to nearest even, and a context that hands out fp32 slices (packed_layer, before or after the slices
were gathered) trains to the same bits as one that does not."""
import pytest
import torch

from paper_1910_02120_b200 import api

pytestmark = pytest.mark.gpu


def _context(dims, S, W, b, batch=32):
    ctx = api.Ist(dims, S, api.IST_BF16, batch)
    ctx.bind_weights([w.clone() for w in W], [v.clone() for v in b])
    return ctx


def _weights(dims, seed=1):
    g = torch.Generator(device="cuda").manual_seed(seed)
    W = [torch.randn(a, b, device="cuda", generator=g) * 0.1 for a, b in zip(dims, dims[1:])]
    return W, [torch.randn(n, device="cuda", generator=g) * 0.1 for n in dims[1:]]


def _bits(x):
    return x.view(torch.int32)


# one entry less and more than a block of the conversion (1024 words), matrices of every move kernel
@pytest.mark.parametrize("dims,S", [([8, 128, 8], 1), ([8, 129, 8], 1), ([33, 31, 70, 9], 3), ([1540, 8189, 8], 3),
                                    ([8, 3100, 1031], 4)])
def test_special_values_come_back(dims, S):
    W, b = _weights(dims)
    special = [0x00000000, 0x80000000, 0x00000001, 0x007fffff, 0x00800000, 0x3f808000, 0x3f818000, 0xbf808000, 0x3f80ffff,
               0x3f807fff, 0x7f7fffff, 0x7f7f8000, 0x7f800000, 0xff800000, 0xff7fffff, 0x80008000]
    vals = torch.tensor([v - 2 ** 32 if v >= 2 ** 31 else v for v in special], dtype=torch.int32, device="cuda")
    for w in W:
        flat = _bits(w.view(-1))
        flat[::3] = vals.repeat(flat[::3].numel() // len(special) + 1)[:flat[::3].numel()]
    for late in (False, True):
        ctx = _context(dims, S, W, b)
        ctx.partition(11)
        want = [[ctx.get_subnet_params(l, s)[0] for s in range(S)] for l in range(1, len(dims))]
        if late:
            for l in range(1, len(dims)):
                m, _ = ctx.packed_layer(l)
                for s in range(S):
                    r, c = want[l - 1][s].shape
                    ld = (-(-dims[l] // (S if l < len(dims) - 1 else 1)) + 7) // 8 * 8
                    assert torch.equal(_bits(m[s][:r * ld].view(r, ld)[:, :c].contiguous()), _bits(want[l - 1][s]))
                    assert torch.equal(_bits(ctx.get_subnet_params(l, s)[0]), _bits(want[l - 1][s]))
        ctx.reassemble()
        ctx.sync_status()
        for w, v in zip(ctx.W, W):
            assert torch.equal(_bits(w), _bits(v))


def test_a_nan_stays_a_nan():
    dims = [16, 64, 8]
    W, b = _weights(dims)
    _bits(W[0].view(-1))[5] = 0x7fffffff                    # rounds up past the exponent unless it is replaced
    _bits(W[0].view(-1))[70] = 0x7f800001                   # its upper half alone is an infinity
    ctx = _context(dims, 2, W, b)
    ctx.partition(3)
    ctx.reassemble()
    assert torch.equal(torch.isnan(ctx.W[0]), torch.isnan(W[0]))


# tiles of 64 and 128 columns on single CTAs, CTA pairs, and widths that leave remainders of each
@pytest.mark.parametrize("dims,S,B", [([64, 512, 16], 4, 128), ([72, 1001, 515, 40], 3, 200), ([256, 2048, 2048, 10], 2, 512),
                                      ([64, 700, 1500], 1, 384)])
def test_handing_out_the_slices_changes_nothing(dims, S, B):
    W, b = _weights(dims, 5)
    for w in W:                                              # some ties of the rounding to bf16, of either kind
        _bits(w.view(-1))[::977] = (_bits(w.view(-1))[::977] & -65536) | 0x8000
    g = torch.Generator(device="cuda").manual_seed(2)
    K = 2
    X = torch.randn(S * K * B, dims[0], device="cuda", generator=g).bfloat16()
    y = torch.randint(dims[-1], (S * K * B,), device="cuda", generator=g, dtype=torch.int32)
    got = []
    for when in ("never", "first", "between"):
        ctx = _context(dims, S, W, b, B)
        if when == "first":
            ctx.packed_layer(1)
        ctx.partition(9)
        if when == "between":
            loss = torch.empty(S, K, device="cuda")
            for k in range(K):                               # one step, the slices handed out, one more
                part = ctx.local_steps(X[k * B:], y[k * B:], 0.05, 1, B, stride_subnet=K * B)
                loss[:, k] = part[:, 0]
                ctx.packed_layer(1)
        else:
            loss = ctx.local_steps(X, y, 0.05, K, B)
        ctx.reassemble()
        ctx.sync_status()
        got.append([loss] + ctx.W + ctx.b)
    for other in got[1:]:
        for p, q in zip(got[0], other):
            assert torch.equal(p, q)


def test_operands_are_rounded_to_even():
    """One row of ones through one layer: z = the operand itself, and the loss of two classes tells it apart.  W = 1 + 2^-8 is
    a tie that rounds down to 1, W = 1 + 3 * 2^-8 one that rounds up to 1 + 2^-6."""
    dims, S = [8, 8, 2], 1
    for value, want in ((1 + 2.0 ** -8, 1.0), (1 + 3 * 2.0 ** -8, 1 + 2.0 ** -6), (1 + 2.0 ** -8 + 2.0 ** -20, 1 + 2.0 ** -7),
                        (1 + 2.0 ** -8 - 2.0 ** -20, 1.0)):
        W = [torch.zeros(8, 8, device="cuda"), torch.zeros(8, 2, device="cuda")]
        W[0][0, 0] = value
        W[1][0, 0] = 1.0
        b = [torch.zeros(8, device="cuda"), torch.zeros(2, device="cuda")]
        X = torch.zeros(1, 8, device="cuda", dtype=torch.bfloat16)
        X[0, 0] = 1
        ctx = _context(dims, S, W, b, 1)
        loss = ctx.round(1, X, torch.zeros(1, device="cuda", dtype=torch.int32), 0.0, 1, 1)
        ctx.sync_status()
        expected = torch.log1p(torch.exp(torch.tensor(-want, dtype=torch.float64)))
        assert abs(float(loss) - float(expected)) <= 1e-6, (value, float(loss), float(expected))
        assert torch.equal(_bits(ctx.W[0]), _bits(W[0]))      # lr = 0: the weight comes back as it was


def _all_kinds(shape, g):
    """Random patterns, half of them with a low half at an edge of the two forms, NaNs among them."""
    n = shape[0] * shape[1]
    high = torch.randint(-2 ** 15, 2 ** 15, (n,), device="cuda", generator=g, dtype=torch.int32)
    low = torch.randint(0, 2 ** 16, (n,), device="cuda", generator=g, dtype=torch.int32)
    edges = torch.tensor([0x7fff, 0x8000, 0x7ffe, 0x8001, 0, 0xffff, 1], dtype=torch.int32, device="cuda")
    low[::2] = edges.repeat(n)[:low[::2].numel()]
    return ((high << 16) | low).view(torch.float32).view(shape)


def _same(p, q):
    nan = torch.isnan(q)
    return torch.equal(torch.isnan(p), nan) and torch.equal(_bits(p.contiguous())[~nan], _bits(q.contiguous())[~nan])


# matrices of every move kernel, odd columns among them
@pytest.mark.parametrize("dims,S", [([8, 128, 8], 1), ([33, 61, 70, 9], 3), ([1540, 8189, 8], 3), ([2048, 4096, 16], 4),
                                    ([8, 3100, 1031], 4)])
def test_every_pattern_is_kept(dims, S):
    g = torch.Generator(device="cuda").manual_seed(6)
    W = [_all_kinds((a, b), g) for a, b in zip(dims, dims[1:])]
    b = [torch.zeros(n, device="cuda") for n in dims[1:]]
    for late in (False, True):
        ctx = _context(dims, S, W, b)
        for seed in (11, 12):                                # the second round finds the first one's tie bits
            ctx.partition(seed)
            parts = [ctx.get_partition(l) for l in range(1, len(dims) - 1)]
            if late and seed == 12:
                ctx.packed_layer(1)
            for s in range(S):
                own = [torch.arange(dims[0], device="cuda")] + [i[o[s]:o[s + 1]].long() for i, o in parts] + [
                    torch.arange(dims[-1], device="cuda")]
                for l in range(1, len(dims)):
                    assert _same(ctx.get_subnet_params(l, s)[0], W[l - 1][own[l - 1]][:, own[l]])
            for w in (ctx.W[0], ctx.W[-1]):                  # every entry of these comes back from a slice
                w.zero_()
            ctx.reassemble()
            ctx.sync_status()
            for w, v in zip(ctx.W, W):
                assert _same(w, v)


def _train(dims, S, B, K, W, b, X, y, lr, when):
    ctx = _context(dims, S, W, b, B)
    if when == "first":
        ctx.packed_layer(1)
    ctx.partition(9)
    if when == "between":
        half = K // 2
        a = ctx.local_steps(X, y, lr, half, B, stride_subnet=K * B)
        ctx.packed_layer(1)
        loss = torch.cat([a, ctx.local_steps(X[half * B:], y[half * B:], lr, K - half, B, stride_subnet=K * B)], 1)
    else:
        loss = ctx.local_steps(X, y, lr, K, B)
    for w in (ctx.W[0], ctx.W[-1]):
        w.zero_()
    ctx.reassemble()
    ctx.sync_status()
    return [loss] + ctx.W + ctx.b


# tiles of 64 and 128 columns on single CTAs, CTA pairs; one master in 2^17 lands on a tie that rounds down in every step
@pytest.mark.parametrize("dims,S,B", [([64, 512, 16], 4, 128), ([1001, 5000, 3001, 77], 6, 200), ([256, 2048, 2048, 10], 2, 512),
                                      ([64, 700, 1500], 1, 384)])
def test_a_long_phase_keeps_every_bit(dims, S, B):
    W, b = _weights(dims, 5)
    for w in W:                                              # and some start on one, of either kind
        _bits(w.view(-1))[::977] = (_bits(w.view(-1))[::977] & -65536) | 0x8000
    g = torch.Generator(device="cuda").manual_seed(2)
    K = 40
    X = torch.randn(S * K * B, dims[0], device="cuda", generator=g)
    X = X.bfloat16() if dims[0] % 8 == 0 else X
    y = torch.randint(dims[-1], (S * K * B,), device="cuda", generator=g, dtype=torch.int32)
    got = [_train(dims, S, B, K, W, b, X, y, 0.002, when) for when in ("never", "first", "between")]
    assert all(bool(torch.isfinite(p).all()) for p in got[0])
    for other in got[1:]:
        for p, q in zip(got[0], other):
            assert torch.equal(p, q)


@pytest.mark.parametrize("dims,S,B", [([16, 100, 8300], 1, 40), ([40, 300, 90], 2, 130), ([40, 300, 90], 2, 30), ([256, 1100, 320], 1, 300)])
def test_updates_keep_ties(dims, S, B):
    """A learning rate of zero: every master is taken apart and joined again.  (The pass over a very wide output layer; updates
    of 128 and 64 columns and of pairs.)"""
    W, b = _weights(dims, 3)
    low = torch.tensor([0x7fff, 0x8000, 0x7ffe, 0x8001], dtype=torch.int32, device="cuda")
    for w in W:
        flat = _bits(w.view(-1))
        flat[:] = (flat & -65536) | low.repeat(flat.numel())[:flat.numel()]
    X = torch.randn(S * B, dims[0], device="cuda").bfloat16()
    y = torch.randint(dims[-1], (S * B,), device="cuda", dtype=torch.int32)
    ctx = _context(dims, S, W, b, B)
    ctx.partition(1)
    for _ in range(2):
        ctx.local_steps(X, y, 0.0, 1, B)
    for w in ctx.W:
        w.zero_()
    ctx.reassemble()
    ctx.sync_status()
    for w, v in zip(ctx.W, W):
        assert torch.equal(_bits(w), _bits(v))
