"""How far an FP32 gradient of the hit-ranking MLP may be from the FP64 one,
parameter by parameter (shared by the CPU and GPU tests)."""
import numpy as np

from oracle import mlp

EPS = 2.0 ** -24


def case(n):
    """Weights, features and labels of a batch of n.  In a large one every sample
    before the last chunk of 256 has features of zero: it adds nothing to the
    gradient of W1, nor to that gradient's bound."""
    rng = np.random.default_rng(n)
    X = rng.normal(size=(n, mlp.N_IN)).astype(np.float32)
    if n > 2000:
        X[:(n - 1) // 256 * 256] = 0.0
    y = (rng.random(n) < 0.5).astype(np.float32)
    return mlp.init_weights(3), X, y


def gradient_bound(w, X, y):
    """A pre-activation is 12 FMAs and a logit 64 more, each rounded once: a logit
    is off by dz <= 77 EPS times the sum of its terms' magnitudes, its sigmoid by a
    quarter of that and by the 8 EPS of its exponential and quotient.  A term of a
    parameter's sum is a product of at most four factors; an activation itself is
    off by 13 EPS of its own terms.  A unit whose pre-activation is within its error
    of zero may or may not count.  Compensated sums, of 256 terms and of the chunks,
    add 4 EPS of the sum of magnitudes.  Returns (bound per parameter, of the loss)."""
    X = X.astype(np.float64)
    n = X.shape[0]
    nw = mlp.N_HID * mlp.N_IN
    W1, b1 = w[:nw].reshape(mlp.N_HID, mlp.N_IN), w[nw:nw + mlp.N_HID]
    w2, b2 = w[nw + mlp.N_HID:nw + 2 * mlp.N_HID], w[-1]
    a = X @ W1.T + b1
    mag = np.abs(X) @ np.abs(W1).T + np.abs(b1)
    da = 13 * EPS * mag
    h, on, unsure = np.maximum(a, 0.0), a > -da, np.abs(a) <= da
    z = h @ w2 + b2
    dz = 77 * EPS * (mag @ np.abs(w2) + np.abs(b2))
    s = 1.0 / (1.0 + np.exp(-z))
    g = np.abs(s - y)
    dg = dz / 4 + 8 * EPS * g + 2 * EPS
    # of d loss / d a_j, and of its sums with x, 1 and (for w2) of g h
    dA = np.where(on, (dg + 8 * EPS * g)[:, None] * np.abs(w2), 0.0) + np.where(unsure, g[:, None] * np.abs(w2), 0.0)
    bW = dA.T @ np.abs(X)
    b_b1 = dA.sum(0)
    b_w2 = (dg + 8 * EPS * g) @ (h + da) + g @ np.where(on, da, 0.0)
    b_b2 = (dg + 8 * EPS * g).sum()
    loss = np.maximum(z, 0.0) - z * y + np.log1p(np.exp(-np.abs(z)))
    return np.concatenate([bW.reshape(-1), b_b1, b_w2, [b_b2]]) / n, (dz + 8 * EPS * (np.abs(z) + loss)).sum() / n
