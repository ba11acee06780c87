"""Partition of all hidden layers in one launch: around the block and cluster sizes, both rules, more
layers than a launch takes, and sizes that go to the whole-GPU launches."""
import numpy as np
import pytest
import torch

from oracle import ist_oracle as O
from paper_1910_02120_b200 import api

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rule", ["balanced", "iid"])
@pytest.mark.parametrize("hidden,S", [((1, 2), 1), ((7, 8, 9), 7), ((1023, 1024, 1025), 3), ((8191, 8193), 5),
                                      ((16384, 16385, 2049), 16), ((40,) * 11, 4), ((700,), 700),
                                      # above 2^14 neurons a layer takes the whole-GPU launches; the second draw mixes both routes
                                      ((16385,), 16), ((16384, 40, 16385, 24), 16)])
def test_partition_and_reassembly(hidden, S, rule):
    dims = [3, *hidden, 5]
    g = torch.Generator(device="cuda").manual_seed(S)
    if len(hidden) < 4 and max(hidden) > 9000:           # keep the middle matrices small enough to hold
        dims = [3, *hidden[:1], *hidden[2:], 5]
    W = [torch.randn(a, b, device="cuda", generator=g) for a, b in zip(dims, dims[1:])]
    b = [torch.randn(n, device="cuda", generator=g) for n in dims[1:]]
    W0, b0 = [w.clone() for w in W], [v.clone() for v in b]
    ctx = api.Ist(dims, S, api.IST_FP32, 4, partition_rule=api.IST_PART_IID if rule == "iid" else api.IST_PART_BALANCED)
    ctx.bind_weights(W, b)
    for seed in (1, 2 ** 63 + 12345):
        ctx.partition(seed)
        want = O.partition(seed, dims, S, rule)
        for l, (idx, off) in enumerate(want, 1):
            got_idx, got_off = ctx.get_partition(l)
            assert np.array_equal(got_off.cpu().numpy(), off), l
            assert np.array_equal(got_idx.cpu().numpy(), idx), l
        for l in range(1, len(dims)):                    # the first and last subnet's slices, values bit for bit
            for s in {0, S - 1}:
                Ws, bs = ctx.get_subnet_params(l, s)
                rows = torch.arange(dims[0], device="cuda") if l == 1 else torch.as_tensor(O.group(want, l - 1, s), device="cuda")
                cols = torch.arange(dims[-1], device="cuda") if l == len(dims) - 1 else torch.as_tensor(O.group(want, l, s), device="cuda")
                assert torch.equal(Ws, W0[l - 1][rows.long()][:, cols.long()]) and torch.equal(bs, b0[l - 1][cols.long()])
        ctx.reassemble()
        ctx.sync_status()
        assert all(torch.equal(x, y) for x, y in zip(W + b, W0 + b0))
