"""Rows that only fill a tile add nothing to the indicator's gradient, whatever
the weights: with an infinite bias the entries it reaches are infinite as in
plain FP64 and the others finite, where a filling row's 0 * inf would make them
NaN. Rows 1 below, at and 1 above whole tiles of 4 and 16 rows.

The infinite output unit saturates every logit, so all labels are 0: each row
has dz = 1 / n, and the finite entries are sums of at most 1025 FP32 terms behind
chains of 25 (1D) and 64 terms: 1200 roundings of 2^-24 of the norm at worst."""
import numpy as np
import pytest

pytestmark = [pytest.mark.gpu, pytest.mark.usefixtures('cuda')]

TOL = 1200 * 2.0 ** -24


def reference(X, w):
    """Gradient for labels 0 in FP64; the hidden ReLUs pass where positive."""
    K, n = X.shape[1], len(X)
    X, w = X.astype(np.float64), w.astype(np.float64)
    W1, b1, W2, b2, w3, b3 = np.split(w, np.cumsum([64 * K, 64, 64 * 64, 64, 64]))
    W1, W2 = W1.reshape(64, K), W2.reshape(64, 64)
    h1 = np.maximum(X @ W1.T + b1, 0.0)
    h2 = np.maximum(h1 @ W2.T + b2, 0.0)
    z = h2 @ w3 + b3
    assert np.all(z == np.inf)
    dz = np.full(n, 1.0 / n)
    d2 = np.where(h2 > 0.0, dz[:, None] * w3, 0.0)
    d1 = np.where(h1 > 0.0, d2 @ W2, 0.0)
    return np.concatenate([(d1.T @ X).ravel(), d1.sum(0), (d2.T @ h1).ravel(), d2.sum(0), dz @ h2, [dz.sum()]])


@pytest.mark.parametrize('n', [1, 3, 4, 5, 511, 512, 513, 1023, 1025, 1040])
def test_filling_rows_add_nothing(n):
    from paper_2508_05020_gb300 import amr
    rng = np.random.default_rng(n)
    K = amr.mlp_k(1)
    X = rng.normal(0.0, 0.3, size=(n, K)).astype(np.float32)
    w = rng.normal(0.0, 0.2, size=64 * K + 64 + 64 * 64 + 64 + 64 + 1).astype(np.float32)
    unit = 64 * K + 64 + 64 * 64 + 7                     # bias of unit 7 of the second layer
    w[unit] = np.inf
    w[unit + 64] = 0.5                                   # its output weight
    loss, g = amr.mlp_grad(1, X, np.zeros(n, dtype=np.float32), 2.5, w)
    want = reference(X, w)
    assert loss == np.inf
    fin = np.isfinite(want)
    assert np.count_nonzero(~fin) == 1 and g[~fin][0] == np.inf
    assert np.all(np.isfinite(g[fin]))
    assert np.linalg.norm(g[fin] - want[fin]) <= TOL * np.linalg.norm(want[fin])
