"""Loss gradient of the learned indicator at the row counts where its kernels
change tile or leave a remainder (4, 8 and 16 rows per tile, clusters of four
blocks, row splits of the first layer's gradient), against plain FP64.

Tolerance: the longest chain of FP32 operations behind an entry is the K sum
of layer 1 (20 + 5), the two 64-term sums of layer 2, and the sum over the
rows (at most 700 terms here in one accumulator): about 900 roundings of
2^-24, 5.4e-5 of the gradient's norm at worst.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

TOL = 900 * 2.0 ** -24


@pytest.fixture(scope='module', autouse=True)
def cuda():
    torch = pytest.importorskip('torch')
    if not torch.cuda.is_available():
        pytest.skip('no CUDA device')
    import __graft_entry__
    __graft_entry__.build()
    torch.cuda.set_device(0)
    yield


def grad64(X, y, pw, w):
    import torch
    K = X.shape[1]
    X, y = torch.from_numpy(X).double(), torch.from_numpy(y).double()
    w = torch.from_numpy(w).double().requires_grad_(True)
    W1, b1, W2, b2, W3, b3 = torch.split(w, [64 * K, 64, 64 * 64, 64, 64, 1])
    h = torch.relu(X @ W1.reshape(64, K).T + b1)
    h = torch.relu(h @ W2.reshape(64, 64).T + b2)
    z = h @ W3 + b3
    sp = torch.nn.functional.softplus
    loss = (pw * y * sp(-z) + (1 - y) * sp(z)).mean()
    loss.backward()
    return float(loss.detach()), w.grad.numpy()


@pytest.mark.parametrize('dim', [1, 2, 3])
@pytest.mark.parametrize('n', [1, 3, 17, 511, 513, 1024, 1025, 2048, 2777])
def test_gradient_matches_fp64(dim, n):
    from paper_2508_05020_gb300 import amr
    rng = np.random.default_rng(100 * dim + n)
    K = amr.mlp_k(dim)
    X = rng.normal(0.0, 0.3, size=(n, K)).astype(np.float32)
    y = (rng.uniform(size=n) < 0.3).astype(np.float32)
    w = rng.normal(0.0, 1.0, size=64 * K + 64 + 64 * 64 + 64 + 64 + 1).astype(np.float32)
    w[:64 * K] *= np.float32(np.sqrt(2.0 / K))
    w[64 * K + 64:] *= np.float32(np.sqrt(2.0 / 64))
    loss, g = amr.mlp_grad(dim, X, y, 2.5, w)
    ref_loss, ref = grad64(X, y, 2.5, w)
    assert abs(loss - ref_loss) <= TOL * abs(ref_loss)
    assert np.linalg.norm(g - ref) <= TOL * np.linalg.norm(ref)
    # every block of the flat layout, so that a small one cannot hide behind W1
    edges = np.cumsum([0, 64 * K, 64, 64 * 64, 64, 64, 1])
    for a, b in zip(edges[:-1], edges[1:]):
        assert np.linalg.norm(g[a:b] - ref[a:b]) <= TOL * max(np.linalg.norm(ref[a:b]), 1e-3 * np.linalg.norm(ref))
