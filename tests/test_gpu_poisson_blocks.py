"""The Poisson solver's block reductions where they can go wrong: fewer cells
than a block's threads, one cell more or fewer than whole blocks, a single
block and many, against the oracle's converged solution (residual 1e-12 on both
sides: the potentials agree to the conditioning times that, bar 1e-9 of the
largest, as in test_gpu_poisson)."""
import numpy as np
import pytest

import oracle as O
import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    import torch
    assert torch.cuda.is_available()
    import __graft_entry__ as ge
    ge.build()
    import paper_2604_12672_gb300 as P
    return P


@pytest.mark.parametrize("n", [(2, 2, 2), (3, 5, 2), (17, 5, 3), (16, 4, 4), (257, 2, 2), (16, 16, 6), (37, 41, 29)])
def test_sizes(P, n):
    xf = [W.random_faces(k, 11 + a) for a, k in enumerate(n)]
    rho = W.lumpy_density(xf, 3)
    kw = dict(lmax=2, criterion="relative", tol=1e-12, max_iter=5000)
    phi, it, res = P.Poisson(xf, **kw).solve(rho)
    ref = O.Poisson(xf, **kw).solve(rho)[0]
    assert res < 1e-12 and it >= 1
    assert np.abs(phi - ref).max() <= 1e-9 * np.abs(ref).max()
