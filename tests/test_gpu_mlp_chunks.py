"""The gradient kernel of the hit-ranking MLP at the edges of its 256-sample
chunks, against the FP64 MLP oracle with the same bfloat16-rounded weights."""
import numpy as np
import pytest
import torch

from oracle import mlp

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 2, 3, 4, 5, 31, 255, 256, 257, 511, 1027, 20001])
def test_gradient_and_step_at_chunk_edges(n):
    """Tolerance: a logit is a chain of 12 + 64 FP32 FMAs, off by at most 76 2^-24
    times the sum of its terms' magnitudes (below 8 here: 4e-5), and the sigmoid's
    slope is at most 1/4; the sum over samples is compensated.  So each term of a
    parameter's gradient is off by at most 1e-5 of |x| (or of |w2 x| in W1)."""
    from paper_1811_04141_gb300 import Context
    from paper_1811_04141_gb300.api import mkf_mlp_grad, mkf_mlp_to_bf16, mkf_mlp_train_step
    ctx = Context(0)
    rng = np.random.default_rng(n)
    # an offset of one float: the features need no alignment
    flat = torch.zeros(n * mlp.N_IN + 1, device="cuda")
    X = rng.normal(size=(n, mlp.N_IN)).astype(np.float32)
    feat = flat[1:].view(n, mlp.N_IN)
    feat.copy_(torch.as_tensor(X))
    y = (rng.random(n) < 0.5).astype(np.float32)
    label = torch.as_tensor(y, device="cuda")
    w = mlp.init_weights(3)
    wd = torch.as_tensor(w, device="cuda", dtype=torch.float32)
    wb = mkf_mlp_to_bf16(ctx, wd)
    g, loss = mkf_mlp_grad(ctx, wb, feat, label)
    lr, gr = mlp.loss_and_grad(mlp.bf16_round(w), X.astype(np.float64), y.astype(np.float64))
    tol = 1e-5 * max(1.0, np.abs(X).max()) * max(1.0, np.abs(w).max()) * 8
    assert np.abs(g.cpu().numpy() - gr).max() <= tol
    assert abs(loss.item() - lr) <= 4e-5 * 8
    # a training step rounds the FP32 weights itself: the same gradient (m = 0.1 g)
    m, v = torch.zeros_like(wd), torch.zeros_like(wd)
    mkf_mlp_train_step(ctx, feat, label, wd, m, v, 1, wb, loss=torch.empty(1, device="cuda"))
    ctx.sync()
    assert torch.equal(m, (1.0 - torch.tensor(0.9, device="cuda")) * g)
    assert torch.equal(wb, mkf_mlp_to_bf16(ctx, wd))
    ctx.close()
