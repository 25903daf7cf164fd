"""The network's loss gradient around the edges of its tiles (64 samples) and of
the grid (456 blocks), against back-propagation in FP64.  Bar: each gradient
entry is a sum over the samples of products that carry ~20 FP32 roundings of
64-term sums of O(1) values (64 x 6e-8 = 4e-6 at worst), added in FP32: 1e-5 of
the sum of the terms' magnitudes."""
import numpy as np
import pytest

from test_gpu_mlp import _bf16_weights, _random_weights

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    import __graft_entry__ as ge
    ge.build()
    import paper_2604_12672_gb300 as P
    return P


@pytest.mark.parametrize("n", [1, 63, 64, 65, 456 * 64, 456 * 64 + 1, 60001])
def test_gradient_at_tile_edges(P, n):
    w = _bf16_weights(_random_weights(5, 0.3)).astype(np.float64)
    W1, b1, W2, b2, W3, b3 = w[:192].reshape(64, 3), w[192:256], w[256:4352].reshape(64, 64), w[4352:4416], w[4416:4480], w[4480]
    r = np.random.default_rng(n)
    x, t = r.uniform(-1, 1, (n, 3)).astype(np.float32), r.uniform(-1, 1, n).astype(np.float32)
    net = P.Mlp(seed=1)
    net.set_weights(w)
    loss, g = net.loss_grad(x, t)
    net.close()
    x64 = x.astype(np.float64)
    h1 = np.tanh(x64 @ W1.T + b1)
    h2 = np.tanh(h1 @ W2.T + b2)
    res = h2 @ W3 + b3 - t
    dy = 2 * res / n
    d2 = dy[:, None] * W3 * (1 - h2 * h2)
    d1 = (d2 @ W2) * (1 - h1 * h1)
    m1 = (np.abs(d2) @ np.abs(W2)) * (1 - h1 * h1)   # magnitudes of d1's terms

    def sums(d1, d2, dy, x, h1, h2):
        return np.concatenate([(d1.T @ x).ravel(), d1.sum(0), (d2.T @ h1).ravel(), d2.sum(0), dy @ h2, [dy.sum()]])

    ref = sums(d1, d2, dy, x64, h1, h2)
    mag = sums(m1, np.abs(d2), np.abs(dy), np.abs(x64), np.abs(h1), np.abs(h2))
    mag = np.maximum(mag, sums(*[np.full_like(a, 2 / n) for a in (d1, d2, dy)], np.abs(x64), np.abs(h1), np.abs(h2)))
    assert abs(loss / np.mean(res * res) - 1) <= 1e-5
    assert (np.abs(g - ref) <= 1e-5 * mag).all()
