"""How the network's loss is summed over many samples: many copies of one
sample have the loss of that sample; a tile's 16 squared residuals of a warp are
added in FP32 (two roundings for equal terms, 1.2e-7), the tiles in FP64.  A
chain of equal terms in FP32 is off by its length times half a unit, 1e-5 here."""
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
