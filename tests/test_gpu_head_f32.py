"""The fp32 path's narrow output layer in one launch (logits, softmax, both deltas) against the oracle."""
import numpy as np
import pytest

from paper_1910_02120_b200 import api, synth
from tests import helpers as H

pytestmark = pytest.mark.gpu


# remainders of 4, 32 and 64 in the neurons, of 8 in the rows, of 4, 8 and 32 in the classes; one of each; the most classes and
# wide layers that are taken, and some that are not
@pytest.mark.parametrize("dims,S,B,K", [
    ([6, 1, 2], 1, 1, 2), ([9, 130, 65, 33], 1, 9, 2), ([20, 63, 64], 1, 8, 2), ([20, 129, 65], 2, 17, 2), ([12, 400, 63], 1, 30, 2),
    ([12, 2022, 10], 1, 12, 2), ([12, 4400, 10], 2, 12, 1), ([33, 600, 41], 5, 100, 3)])
def test_round_matches_oracle(dims, S, B, K):
    w = synth.Workload("h", tuple(dims), S=S, B=B, K=K, rounds=1, precision="fp32", x_dist="normal", lr=0.1, seed=5)
    W, b, data = H.make_problem(w, bias_scale=0.1)
    o, _, olosses = H.oracle_round(w, W, b, data, 9)
    _, Wd, bd, _, losses = H.gpu_round(w, W, b, data, 9)
    assert np.max(np.abs(losses - olosses)) <= 1e-4 * np.abs(olosses).max()
    for l in range(len(W)):
        H.assert_close(Wd[l], o.W[l], 1e-4, f"W_{l + 1}")
        H.assert_close(bd[l], o.b[l], 1e-4, f"b_{l + 1}")
        # fp32 weights hold an update to 2^-24 of a weight, and updates are 2^-12 of the weights or more
        upd, ref = Wd[l].astype(np.float64) - W[l], o.W[l] - W[l]
        assert np.linalg.norm(upd - ref) <= 1e-3 * np.linalg.norm(ref)


def test_a_label_outside_the_classes_is_reported():
    w = synth.Workload("h", (8, 16, 5), S=2, B=6, K=1, rounds=1, precision="fp32", x_dist="normal", lr=0.1, seed=5)
    W, b, data = H.make_problem(w)
    ctx, _, _ = H.gpu_context(w, W, b)
    X, y = H.gpu_inputs(w, data)
    y[3] = 5
    ctx.partition(1)
    ctx.local_steps(X, y, w.lr, 1, w.B)
    with pytest.raises(api.IstError):
        ctx.sync_status()
