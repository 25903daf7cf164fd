"""How the network's loss and gradient are summed over many samples.

Loss: many copies of one sample have the loss of that sample; a tile's 16
squared residuals of a warp are added in FP32 (two roundings for equal terms,
1.2e-7), the tiles in FP64.  A chain of equal terms in FP32 is off by its length
times half a unit, 1e-5 here.

Gradient: 456 blocks add to an entry one after another in FP32, each rounding
2^-24 / sqrt(12) of the sum so far, and the sum grows evenly: sqrt(456 / 3)
times 1.7e-8 = 2.1e-7 of the entry, twice that for the sums inside the blocks."""
import numpy as np
import pytest

from test_gpu_mlp import _bf16_weights, _random_weights

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def net():
    import __graft_entry__ as ge
    ge.build()
    import paper_2604_12672_gb300 as P
    m = P.Mlp(seed=1)
    m.set_weights(_bf16_weights(_random_weights(5, 0.3)).astype(np.float64))
    yield m
    m.close()


@pytest.mark.parametrize("seed", [0, 1, 2, 3])
def test_loss_of_equal_samples(net, seed):
    r = np.random.default_rng(seed)
    x, t = r.uniform(-1, 1, (1, 3)).astype(np.float32), r.uniform(-1, 1, 1).astype(np.float32)
    one = net.loss_grad(x, t)[0]
    many = net.loss_grad(np.repeat(x, 1 << 22, 0), np.repeat(t, 1 << 22))[0]
    assert abs(many / one - 1) <= 2e-7


@pytest.mark.parametrize("n", [65536, 300000])
def test_gradient_rms(net, n):
    w = net.get_weights().astype(np.float64)
    W1, b1, W2, b2, W3, b3 = w[:192].reshape(64, 3), w[192:256], w[256:4352].reshape(64, 64), w[4352:4416], w[4416:4480], w[4480]
    r = np.random.default_rng(n)
    x, t = r.uniform(-1, 1, (n, 3)).astype(np.float32), r.uniform(-1, 1, n).astype(np.float32)
    g = net.loss_grad(x, t)[1]
    x = x.astype(np.float64)
    h1 = np.tanh(x @ W1.T + b1)
    h2 = np.tanh(h1 @ W2.T + b2)
    dy = 2 * (h2 @ W3 + b3 - t) / n
    d2 = dy[:, None] * W3 * (1 - h2 * h2)
    d1 = (d2 @ W2) * (1 - h1 * h1)
    ref = np.concatenate([(d1.T @ x).ravel(), d1.sum(0), (d2.T @ h1).ravel(), d2.sum(0), dy @ h2, [dy.sum()]])
    assert np.linalg.norm(g - ref) <= 4.2e-7 * np.linalg.norm(ref)
