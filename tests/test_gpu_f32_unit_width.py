"""fp32 rounds with a single input feature: the rows of X have unit stride in both directions, beside other
layers' operands that have it in one (the weight updates of all layers are one launch)."""
import pytest

from paper_1910_02120_b200 import synth
from tests import helpers as H

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims,S", [((1, 16, 3), 1), ((1, 16, 16, 3), 2), ((1, 1, 3), 1), ((1, 9, 1, 5, 2), 1), ((1, 4, 1), 4)])
@pytest.mark.parametrize("B", [1, 4, 70])          # short contractions, and beyond 64 rows the tensor-core kernel
def test_round(dims, S, B):
    w = synth.Workload("unit", dims, S=S, B=B, K=3, rounds=1, precision="fp32", x_dist="normal", lr=0.05, seed=B)
    W, b, data = H.make_problem(w)
    o, _, oloss = H.oracle_round(w, W, b, data, 5)
    _, gW, gb, _, gloss = H.gpu_round(w, W, b, data, 5)
    H.assert_close(gloss, oloss, 1e-4, "losses")
    for l in range(len(W)):
        H.assert_close(gW[l], o.W[l], 1e-4, f"W_{l + 1}")
        H.assert_close(gb[l], o.b[l], 1e-4, f"b_{l + 1}")
