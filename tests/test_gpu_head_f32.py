"""The fp32 path's narrow output layer in one launch (logits, softmax, both deltas) against the oracle."""
import numpy as np
import pytest
import torch

from oracle import ist_oracle as O
from paper_1910_02120_b200 import api, synth
from tests import helpers as H

pytestmark = pytest.mark.gpu


def _check(w, taken, norm_eps=None):
    W, b, data = H.make_problem(w, bias_scale=0.1)
    o, _, olosses = H.oracle_round(w, W, b, data, 9, norm_eps=norm_eps)
    ctx, Wd, bd = H.gpu_context(w, W, b)
    if norm_eps is not None:
        ctx.enable_normalization(norm_eps)
    ctx.profile(True)
    X, y = H.gpu_inputs(w, data)
    losses = ctx.round(9, X, y, w.lr, w.K, w.B).cpu().numpy()
    ctx.sync_status()
    prof, t = ctx.profile_read(), len(W)
    # one launch from the activations to both deltas, or one more product on either side of the softmax
    assert prof["loss"][0] == w.K and prof["dx"][0] == w.K * (t - 1 - taken)
    tol = 1e-4 if norm_eps is None else 2e-4                  # standardisation multiplies rounding errors by 1 / sigma
    assert np.max(np.abs(losses - olosses)) <= tol * np.abs(olosses).max()
    for l in range(t):
        H.assert_close(Wd[l].cpu().numpy(), o.W[l], tol, f"W_{l + 1}")
        H.assert_close(bd[l].cpu().numpy(), o.b[l], tol, f"b_{l + 1}")
        # fp32 weights hold an update to 2^-24 of a weight, and updates are 2^-12 of the weights or more
        upd, ref = Wd[l].cpu().numpy().astype(np.float64) - W[l], o.W[l] - W[l]
        assert np.linalg.norm(upd - ref) <= 1e-3 * np.linalg.norm(ref)


# remainders of 4, 32 and 64 in the neurons, of 8 in the rows, of 4, 8 and 32 in the classes; one of each; the most classes and
# wide layers that are taken, and some that are not
@pytest.mark.parametrize("dims,S,B,K,taken", [
    ([6, 1, 2], 1, 1, 2, True), ([9, 130, 65, 33], 1, 9, 2, True), ([20, 63, 64], 1, 8, 2, True), ([20, 129, 65], 2, 17, 2, False),
    ([12, 400, 63], 1, 30, 2, True), ([12, 2022, 10], 1, 12, 2, False), ([12, 1700, 10], 1, 12, 2, True),
    ([12, 4400, 10], 2, 12, 1, False), ([33, 600, 41], 5, 100, 3, True)])
def test_round_matches_oracle(dims, S, B, K, taken):
    w = synth.Workload("h", tuple(dims), S=S, B=B, K=K, rounds=1, precision="fp32", x_dist="normal", lr=0.1, seed=5)
    _check(w, taken)


# what the launches around it make of its two deltas and its activations
@pytest.mark.parametrize("kind", ["norm", "csr"])
def test_beside_standardisation_and_sparse_rows(kind):
    csr = dict(x_dist="csr", csr_mean_nnz=8.0) if kind == "csr" else dict(x_dist="normal")
    w = synth.Workload("h", (200, 90, 70, 12), S=2, B=40, K=3, rounds=1, precision="fp32", lr=0.05, seed=5, **csr)
    _check(w, True, norm_eps=1e-5 if kind == "norm" else None)


def test_beside_the_input_gradient():
    w = synth.Workload("h", (24, 90, 70, 12), S=2, B=40, K=2, rounds=1, precision="fp32", x_dist="normal", lr=0.05, seed=5)
    W, b, data = H.make_problem(w, bias_scale=0.1)
    o = O.IstOracle(w.layer_dims, w.S)
    o.bind_weights(W, b)
    o.partition(9)
    _, odx = o.local_steps_dx(data.X, data.y, w.lr, w.K)
    ctx, _, _ = H.gpu_context(w, W, b)
    ctx.profile(True)
    X, y = H.gpu_inputs(w, data)
    dx = torch.empty(X.shape[0], w.layer_dims[0], device="cuda")
    ctx.partition(9)
    ctx.local_steps(X, y, w.lr, w.K, w.B, dx_out=dx)
    ctx.sync_status()
    assert ctx.profile_read()["dx"][0] == w.K * 2             # the middle layer's delta and the input's gradient
    H.assert_close(dx.cpu().numpy().reshape(odx.shape), odx, 1e-4, "dX")


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
