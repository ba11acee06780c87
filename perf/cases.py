"""The work a user of this library has it do, as measurable cases: whole training rounds (partition,
K local steps of all subnets, reassemble), rounds driven one step at a time by a trunk in front of
the partitioned layers, and full-width evaluation of the reassembled network.

A case is a dict of plain values:
  call       "round": one call chain partition -> local_steps(K) -> reassemble;
             "trunk": the same round with K calls of one step each, every call returning the
                      gradient with respect to its input rows;
             "eval":  mean loss and number of correct rows of the bound full network
  dims       layer widths N_0-...-N_t          subnets    S
  batch      rows per subnet and step (for "eval": the context's chunk of rows)
  steps      local steps K                     rows       rows of an evaluation
  precision  operand type of the local steps   x          "f32" / "bf16" dense rows or "csr"
  nnz        mean nonzeros of a CSR row        norm       batch standardisation of the hidden layers
  rule       "balanced" or "iid" assignment    lr         learning rate

Shapes, batch sizes and learning rates come from the workloads of paper_1910_02120_b200.synth, its
two example programs (teacher_student, trunk_head) and the tests.
"""
import math

import torch

from paper_1910_02120_b200 import api


def _case(name, call, dims, subnets, batch, steps=0, rows=0, precision="bf16", x="bf16", nnz=0, norm=False,
          rule="balanced", lr=0.01):
    return {"name": name, "call": call, "dims": dims, "subnets": subnets, "batch": batch, "steps": steps, "rows": rows,
            "precision": precision, "x": x, "nnz": nnz, "norm": norm, "rule": rule, "lr": lr}


def listed():
    return [
        # the partitioned head of a larger network: one local step per call, the trunk waits for dX each time
        _case("trunk-fp32", "trunk", "64-256-256-10", 4, 64, 10, precision="fp32", x="f32", lr=0.3),
        # a small classifier in full precision
        _case("tiny-fp32", "round", "784-1024-10", 2, 128, 10, precision="fp32", x="f32"),
        # a small network with the paper's batch standardisation, many short rounds
        _case("teacher-norm-bf16", "round", "64-512-512-10", 4, 64, 10, norm=True, lr=0.05),
        # speech-command network: a long local phase on subnets that stay in L2
        _case("speech-bf16", "round", "1024-4096-4096-35", 4, 256, 50),
        # the same network in full precision
        _case("speech-fp32", "round", "1024-4096-4096-35", 4, 256, 10, precision="fp32", x="f32"),
        # nothing divides anything, subnets of unequal size, rows handed over as fp32
        _case("ragged-iid-bf16", "round", "1001-5000-3001-77", 6, 200, 8, x="f32", rule="iid"),
        # medium width with a hundred classes
        _case("medium-bf16", "round", "1024-8192-8192-100", 4, 512, 10),
        # the wide pixel network: the library's main workload
        _case("pixels-bf16", "round", "3072-16384-16384-10", 8, 512, 20),
        # a very wide network re-partitioned after every step: moving slices is most of the round
        _case("wide-one-step-bf16", "round", "1024-32768-32768-100", 8, 512, 1),
        # extreme classification: sparse features, 670,091 classes
        _case("extreme-csr-bf16", "round", "135909-1024-670091", 8, 256, 10, x="csr", nnz=75),
        # scoring the reassembled network between rounds
        _case("eval-pixels", "eval", "3072-16384-16384-10", 8, 512, rows=4096, x="f32"),
        _case("eval-extreme-csr", "eval", "135909-1024-670091", 8, 256, rows=1024, x="csr", nnz=75),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _propose(rng):
    kind = rng.choice(["round-bf16", "round-bf16", "round-bf16", "round-fp32", "csr", "trunk", "eval", "eval-csr"])
    multiple = rng.choice([1, 8, 64])                  # odd widths, padded rows, whole tiles

    def width(lo, hi):
        return max(lo, _log(rng, lo, hi) // multiple * multiple)

    S = _log(rng, 1, 16)
    hidden = rng.choice([1, 2, 2, 2, 3])
    classes = _log(rng, 5, 1000)
    if kind == "csr" or kind == "eval-csr":
        dims = [_log(rng, 5000, 135909), width(128, 2048), _log(rng, 1000, 670091)]
    else:
        top = 32768 if kind == "round-bf16" else 16384 if kind == "eval" else 4096
        dims = [width(32, 3072)] + [width(16 * S, top) for _ in range(hidden)] + [classes]
    c = {"call": "round", "dims": "-".join(str(d) for d in dims), "subnets": S, "batch": _log(rng, 24, 640),
         "steps": _log(rng, 1, 50), "rows": 0, "precision": "bf16", "x": "bf16", "nnz": 0, "norm": False,
         "rule": "balanced", "lr": 0.01}
    bf16_rows = dims[0] % 8 == 0
    if kind == "round-bf16":
        c["x"] = "bf16" if bf16_rows and rng.random() < 0.8 else "f32"
        c["norm"] = rng.random() < 0.2
        c["rule"] = "iid" if rng.random() < 0.2 else "balanced"
    elif kind == "round-fp32":
        c.update(precision="fp32", x="f32", norm=rng.random() < 0.2, steps=_log(rng, 1, 20))
    elif kind == "csr":
        c.update(x="csr", nnz=_log(rng, 10, 100), batch=_log(rng, 32, 256), steps=_log(rng, 1, 10),
                 precision=rng.choice(["bf16", "bf16", "bf16", "fp32"]))
        if c["precision"] == "fp32":                   # the fp32 path is for networks of moderate width
            dims[2] = _log(rng, 1000, 20000)
            c["dims"] = "-".join(str(d) for d in dims)
    elif kind == "trunk":
        c.update(call="trunk", steps=_log(rng, 1, 10), batch=_log(rng, 16, 256))
        dims[0] = max(16, dims[0] // 16 * 16)
        c["dims"] = "-".join(str(d) for d in dims)
        c.update(rng.choice([{"precision": "fp32", "x": "f32"}, {"precision": "bf16", "x": "bf16"}]))
    else:
        c.update(call="eval", rows=_log(rng, 64, 8192), steps=0, x="f32")
        if kind == "eval-csr":
            c.update(x="csr", nnz=_log(rng, 10, 100), rows=_log(rng, 64, 1024), batch=_log(rng, 32, 256))
    return c


def _cost(c):
    """A rough time in seconds, by which draw() stays at or below the listed cases."""
    w = work(c)
    full = _full_weights(c)
    per_flop = 1 / 20e12 if c["call"] == "eval" or c["precision"] == "fp32" else 1 / 400e12
    owned = sum(a for a, _ in _slices(c))
    return full * 12 / 4e12 + max(1, c["steps"]) * (owned * 12 / 4e12 + 1e-4) + w["flops"] * per_flop


def draw(rng):
    most = {True: max(_cost(c) for c in listed() if c["call"] == "eval" or c["precision"] == "fp32"),
            False: max(_cost(c) for c in listed())}
    largest = max(work(c)["flops"] for c in listed())
    while True:
        c = _propose(rng)
        if _cost(c) <= most[c["call"] == "eval" or c["precision"] == "fp32"] and work(c)["flops"] <= largest:
            return c


def _dims(case):
    return [int(d) for d in case["dims"].split("-")]


def _full_weights(case):
    d = _dims(case)
    return sum(a * b for a, b in zip(d, d[1:]))


def _slices(case):
    """Per layer: (weights all subnets own, weights a step really touches)."""
    d, S = _dims(case), case["subnets"]
    t = len(d) - 1
    out = []
    for l in range(1, t + 1):
        n = d[l - 1] * d[l]
        if 1 < l < t:
            n //= S
        out.append((n, n))
    if case["x"] == "csr":                             # distinct columns of the rows that are read
        rows = max(case["rows"], case["batch"] * max(1, case["steps"]))
        seen = d[0] * (1.0 - math.exp(-rows * case["nnz"] / d[0]))
        out[0] = (out[0][0], int(seen) * d[1])
    return out


def work(case):
    d, S, B, K = _dims(case), case["subnets"], case["batch"], case["steps"]
    row_bytes = 8 * case["nnz"] if case["x"] == "csr" else d[0] * (2 if case["x"] == "bf16" else 4)
    if case["call"] == "eval":
        n = case["rows"]
        first = case["nnz"] * d[1] if case["x"] == "csr" else d[0] * d[1]
        rest = sum(a * b for a, b in zip(d[1:], d[2:]))
        read = (_slices(case)[0][1] if case["x"] == "csr" else d[0] * d[1]) + rest
        return {"bytes": 4 * read + n * (row_bytes + 4), "flops": 2 * n * (first + rest)}
    # every owned weight is read once and written once; each row goes forward, back and into the update
    per_row = 0
    for l, (owned, _) in enumerate(_slices(case), 1):
        n = owned // S
        if l == 1:
            per_row += 2 * (case["nnz"] * (d[1] // S) if case["x"] == "csr" else n)
            per_row += n if case["call"] == "trunk" else 0
        else:
            per_row += 3 * n
    io = row_bytes + 4 + (4 * d[0] if case["call"] == "trunk" else 0)
    return {"bytes": 8 * sum(touched for _, touched in _slices(case)) + S * K * B * io, "flops": 2 * S * K * B * per_row}


def tolerance(case):
    # Four times what a round differs by from the same round with its sums in 64 bits (and the roundings to
    # bf16 where the path has them), over the listed cases and twenty drawn ones: fp32 at most 9e-7 in the
    # 2-norm and 2.1e-4 in one value (a ReLU that flips), evaluation 3.2e-8; bf16 3.5e-4 and 7.7e-3.
    if case["call"] == "eval" or case["precision"] == "fp32":
        return {"rel": 1e-5, "max": 1e-3}
    return {"rel": 1.5e-3, "max": 3e-2}


def _csr_rows(g, n, n0, mean):
    """Rows of Poisson(mean) (at least one) distinct ascending columns, values |N(0, 1)|."""
    counts = torch.poisson(torch.full((n,), float(mean), device="cuda"), generator=g).clamp_(1, n0).long()
    row = torch.repeat_interleave(torch.arange(n, device="cuda"), counts)
    key = torch.unique(row * n0 + torch.randint(n0, (row.numel(),), device="cuda", generator=g))
    row_ptr = torch.zeros(n + 1, dtype=torch.int32, device="cuda")
    row_ptr[1:] = torch.cumsum(torch.bincount(key // n0, minlength=n), 0)
    return row_ptr, (key % n0).int(), torch.randn(key.numel(), device="cuda", generator=g).abs_()


def _inputs(case, seed):
    d, S, B = _dims(case), case["subnets"], case["batch"]
    g = torch.Generator(device="cuda").manual_seed(seed)
    W, b = [], []
    for fan_in, fan_out in zip(d, d[1:]):
        bound = math.sqrt(6.0 / fan_in)
        W.append(torch.empty(fan_in, fan_out, device="cuda").uniform_(-bound, bound, generator=g))
        b.append(torch.empty(fan_out, device="cuda").uniform_(-0.1, 0.1, generator=g))
    n = case["rows"] or S * case["steps"] * B
    if case["x"] == "csr":
        X = _csr_rows(g, n, d[0], case["nnz"])
    else:
        X = torch.randn(n, d[0], device="cuda", generator=g)
        X = X.to(torch.bfloat16) if case["x"] == "bf16" else X
    y = torch.randint(d[-1], (n,), device="cuda", generator=g, dtype=torch.int32)
    return W, b, X, y


def prepare(case, seed):
    d, S, B = _dims(case), case["subnets"], case["batch"]
    W, b, X, y = _inputs(case, seed)
    ctx = api.Ist(d, S, api.IST_BF16 if case["precision"] == "bf16" else api.IST_FP32, B,
                  input_is_csr=case["x"] == "csr",
                  partition_rule=api.IST_PART_IID if case["rule"] == "iid" else api.IST_PART_BALANCED)
    ctx.bind_weights(W, b)
    if case["norm"]:
        ctx.enable_normalization(1e-5)
    return {"case": case, "ctx": ctx, "X": X, "y": y, "round": seed * 7919}


def run(state):
    case, ctx, X, y = state["case"], state["ctx"], state["X"], state["y"]
    B, K, lr = case["batch"], case["steps"], case["lr"]
    if case["call"] == "eval":
        return ctx.eval(X, y, case["rows"])
    state["round"] += 1                                # every round draws a new partition
    if case["call"] == "round":
        loss = ctx.round(state["round"], X, y, lr, K, B)
        return {"loss": loss, "W": ctx.W, "b": ctx.b}
    ctx.partition(state["round"])
    rows = case["subnets"] * B                         # one call per step: rows [S][B] of step k
    losses, grads = [], []
    for k in range(K):
        dx = torch.empty(rows, X.shape[1], device="cuda")
        losses.append(ctx.local_steps(X[k * rows:(k + 1) * rows], y[k * rows:(k + 1) * rows], lr, 1, B, dx_out=dx))
        grads.append(dx)
    ctx.reassemble()
    return {"loss": losses, "dx": grads, "W": ctx.W, "b": ctx.b}


# ---- the same in 64 bits, with torch alone ------------------------------------------------------

def _splitmix64(state, count):
    """Outputs 1..count of SplitMix64 (Steele, Lea, Flood 2014) from `state`, as int64 bit patterns."""
    def signed(v):
        v &= 2 ** 64 - 1
        return v - 2 ** 64 if v >= 2 ** 63 else v

    def shifted(v, k):                                 # logical shift right
        return (v >> k) & (2 ** (64 - k) - 1)

    z = torch.arange(1, count + 1, device="cuda") * signed(0x9E3779B97F4A7C15) + signed(state)
    z = (z ^ shifted(z, 30)) * signed(0xBF58476D1CE4E5B9)
    z = (z ^ shifted(z, 27)) * signed(0x94D049BB133111EB)
    return z ^ shifted(z, 31)


def _groups(case, round_seed):
    """Per hidden layer the S index sets of the partition that `round_seed` draws."""
    S, out = case["subnets"], []
    for l, n in enumerate(_dims(case)[1:-1], 1):
        key = _splitmix64(int(_splitmix64(round_seed, l)[-1]), n)
        if case["rule"] == "iid":                      # floor(key * S / 2^64) of the unsigned key
            high, low = (key >> 32) & 0xFFFFFFFF, key & 0xFFFFFFFF
            which = (high * S + ((low * S) >> 32)) >> 32
        else:                                          # equal shares of the unsigned order
            which = torch.empty(n, dtype=torch.int64, device="cuda")
            sizes = torch.tensor([n // S + (s < n % S) for s in range(S)], device="cuda")
            order = torch.sort(key ^ -2 ** 63, stable=True).indices
            which[order] = torch.repeat_interleave(torch.arange(S, device="cuda"), sizes)
        out.append([torch.nonzero(which == s).flatten() for s in range(S)])
    return out


class _Rows:
    """Rows r0 .. r0 + n - 1 of the inputs: products with a first-layer matrix and its gradient."""

    def __init__(self, X, r0, n):
        if isinstance(X, tuple):
            row_ptr, col, val = X
            lo, hi = int(row_ptr[r0]), int(row_ptr[r0 + n])
            counts = (row_ptr[r0 + 1:r0 + n + 1] - row_ptr[r0:r0 + n]).long()
            row = torch.repeat_interleave(torch.arange(n, device="cuda"), counts)
            self.csr, self.n = (row, col[lo:hi].long(), val[lo:hi].double()[:, None]), n
        else:
            self.csr, self.x = None, X[r0:r0 + n].double()

    def times(self, W):
        if self.csr is None:
            return self.x @ W
        row, col, val = self.csr
        return torch.zeros(self.n, W.shape[1], dtype=W.dtype, device="cuda").index_add_(0, row, W[col] * val)

    def descend(self, W, delta, lr):
        if self.csr is None:
            W.addmm_(self.x.T, delta, alpha=-lr)
        else:
            row, col, val = self.csr
            W.index_add_(0, col, delta[row] * val, alpha=-lr)


def _step(case, W, b, x, y):
    """One SGD step of one subnet (W, b are changed): the mean loss and d(loss)/d(x) where it is asked for."""
    t, B, a, unit, scale, z = len(W), case["batch"], [], [], [], None
    for l in range(t):
        z = (x.times(W[0]) if l == 0 else a[-1] @ W[l]) + b[l]
        if l + 1 < t:
            if case["norm"]:
                centred = z - z.mean(0)
                scale.append(torch.rsqrt((centred ** 2).mean(0) + 1e-5))
                z = centred * scale[-1]
                unit.append(z)
            a.append(z.clamp_min(0))
    at = torch.arange(B, device="cuda")
    logp = torch.log_softmax(z, 1)
    loss = -logp[at, y].mean()
    delta = torch.exp(logp)
    delta[at, y] -= 1
    delta /= B
    lr, dx = case["lr"], None
    for l in range(t - 1, -1, -1):
        below = delta @ W[l].T if l > 0 or case["call"] == "trunk" else None
        b[l] -= lr * delta.sum(0)
        if l == 0:
            dx = below
            x.descend(W[0], delta, lr)
            break
        W[l].addmm_(a[l - 1].T, delta, alpha=-lr)
        delta = below * (a[l - 1] > 0)
        if case["norm"]:
            zh = unit[l - 1]
            delta = scale[l - 1] * (delta - delta.mean(0) - zh * (delta * zh).mean(0))
    return loss, dx


def exact(case, seed):
    W, b, X, y = _inputs(case, seed)
    y, S, B, K = y.long(), case["subnets"], case["batch"], case["steps"]
    if case["call"] == "eval":
        loss, hits = 0.0, 0
        for r0 in range(0, case["rows"], B):
            n = min(B, case["rows"] - r0)
            z = _Rows(X, r0, n).times(W[0].double()) + b[0]
            for Wl, bl in zip(W[1:], b[1:]):
                z = z.clamp_min(0) @ Wl.double() + bl
            labels = y[r0:r0 + n]
            loss = loss - torch.log_softmax(z, 1)[torch.arange(n, device="cuda"), labels].sum()
            hits = hits + (z.argmax(1) == labels).sum()
        return (loss / case["rows"]).reshape(1), hits.reshape(1)
    t, groups = len(W), _groups(case, seed * 7919 + 1)
    W, b = [w.double() for w in W], [v.double() for v in b]
    out_bias = torch.zeros_like(b[-1])
    losses = torch.empty(S, K, dtype=torch.float64, device="cuda")
    grads = [torch.empty(S * B, _dims(case)[0], dtype=torch.float64, device="cuda") for _ in range(K)] \
        if case["call"] == "trunk" else None
    for s in range(S):
        rows = [slice(None)] + [g[s][:, None] for g in groups[:-1]] + [groups[-1][s]]
        cols = [g[s] for g in groups] + [slice(None)]
        Ws = [W[l][rows[l], cols[l]].clone() for l in range(t)]
        bs = [b[l][cols[l]].clone() for l in range(t)]
        for k in range(K):                             # rows [S][K][B] of a round, [K][S][B] with a trunk
            r0 = (k * S + s) * B if grads is not None else (s * K + k) * B
            losses[s, k], dx = _step(case, Ws, bs, _Rows(X, r0, B), y[r0:r0 + B])
            if grads is not None:
                grads[k][s * B:(s + 1) * B] = dx
        for l in range(t):
            W[l][rows[l], cols[l]] = Ws[l]
            if l + 1 < t:
                b[l][cols[l]] = bs[l]
        out_bias += bs[-1] / S
    b[-1] = out_bias
    if grads is None:
        return {"loss": losses, "W": W, "b": b}
    return {"loss": [losses[:, k:k + 1] for k in range(K)], "dx": grads, "W": W, "b": b}
