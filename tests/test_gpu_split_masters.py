"""Masters kept as bf16 operand and low half: every value that no step has changed comes back bit for bit, the operand
is the master rounded to nearest even, and a context that hands out fp32 slices (packed_layer, before or after the slices
were gathered) trains to the same values as one that does not."""
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
            # a tie is kept 2^-24 off in one form: 2^-24 / sqrt(977) over a matrix; its products move sums by less
            # than their own rounding, so a ReLU that flips is not to be expected
            assert float((p - q).norm()) <= 1e-7 * float(q.norm())


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
