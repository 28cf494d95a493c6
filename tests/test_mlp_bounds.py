"""The bounds of tests/mlp_bounds.py are small enough to see one lost sample."""
import numpy as np
import pytest

from oracle import mlp
from tests.mlp_bounds import case, gradient_bound

SIZES = [2, 5, 31, 255, 256, 257, 511, 1027, 4097, 20001]


@pytest.mark.parametrize("n", SIZES)
def test_a_lost_sample_exceeds_the_bound(n):
    w, X, y = case(n)
    wr = mlp.bf16_round(w).astype(np.float64)
    loss, g = mlp.loss_and_grad(wr, X.astype(np.float64), y.astype(np.float64))
    bound, dl = gradient_bound(wr, X, y)
    # the last sample left out of the sums (which are still divided by n)
    l1, g1 = mlp.loss_and_grad(wr, X[:-1].astype(np.float64), y[:-1].astype(np.float64))
    f = (n - 1) / n
    d = np.abs(g1 * f - g)
    nw = mlp.N_HID * mlp.N_IN
    groups = [(0, nw)] if n > 2000 else [(0, nw), (nw, nw + 64), (nw + 64, nw + 128), (nw + 128, nw + 129)]
    for lo, hi in groups:
        assert (d[lo:hi] > 2.0 * bound[lo:hi]).any(), lo
    assert n > 2000 or abs(l1 * f - loss) > 2.0 * dl
