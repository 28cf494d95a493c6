"""The gradient kernel of the hit-ranking MLP at the edges of its 256-sample
chunks, every parameter within its own rounding bound of the FP64 oracle (a
lost sample is beyond it, see test_mlp_bounds.py)."""
import numpy as np
import pytest
import torch

from oracle import mlp
from tests.mlp_bounds import case, gradient_bound
from tests.test_mlp_bounds import SIZES

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1] + SIZES)
def test_every_parameter_within_its_bound(n):
    from paper_1811_04141_gb300 import Context
    from paper_1811_04141_gb300.api import mkf_mlp_grad, mkf_mlp_to_bf16
    ctx = Context(0)
    w, X, y = case(n)
    wr = mlp.bf16_round(w).astype(np.float64)
    wb = mkf_mlp_to_bf16(ctx, torch.as_tensor(w, device="cuda", dtype=torch.float32))
    g, loss = mkf_mlp_grad(ctx, wb, torch.as_tensor(X, device="cuda"), torch.as_tensor(y, device="cuda"))
    ctx.sync()
    want_loss, want = mlp.loss_and_grad(wr, X.astype(np.float64), y.astype(np.float64))
    bound, dl = gradient_bound(wr, X, y)
    assert (np.abs(g.cpu().numpy() - want) <= bound).all()
    assert abs(loss.item() - want_loss) <= dl
    ctx.close()
