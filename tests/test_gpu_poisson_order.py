"""The order in which the Poisson solver adds up its inner products: BiCGSTAB's
iteration count moves by a tenth with the rounding of these sums, so a change of
order shows as another count.  The counts are those of the fixed order (shuffle
trees over a warp's lanes, over the warps of a block, 32 interleaved chains over
the blocks' partials), on grids of 16 to 608 blocks, whole and partial last
ones; the solver is deterministic."""
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    import __graft_entry__ as ge
    ge.build()
    import paper_2604_12672_gb300 as P
    return P


@pytest.mark.parametrize("n, counts", [((16, 16, 16), (70, 71, 72)), ((20, 24, 28), (104, 122, 117)),
                                       ((32, 32, 32), (137, 139, 138)), ((48, 48, 48), (207, 218, 231)),
                                       ((80, 80, 80), (344, 342, 389))])
def test_counts(P, n, counts):
    xf = [W.random_faces(k, 11 + a) for a, k in enumerate(n)]
    s = P.Poisson(xf, lmax=2, criterion="relative", tol=1e-10, max_iter=5000)
    got = tuple(s.solve(W.lumpy_density(xf, seed))[1] for seed in (3, 4, 5))
    s.close()
    assert got == counts


def test_stretched_sphere(P):
    xf = [W.stretched_faces(128)] * 3
    s = P.Poisson(xf, G=1.0, lmax=0, criterion="absolute", tol=1e-10, max_iter=20000)
    it = s.solve(W.sphere_density(xf))[1]
    s.close()
    assert it == 356
