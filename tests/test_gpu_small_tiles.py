"""The tile kernel's form for grids of at most one tile per SM (152: one face
per thread, the raw flags dilated in the tile) on both sides of that line,
against the per-direction kernels with their own dilation passes: the mixed
form's bar, 1e-5 relative L1 of the deviations.  The flattening threshold is
set low enough that part of the cells is flagged."""
import numpy as np
import pytest

import workloads as W
from test_gpu_mixed import deviation_l1

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    import __graft_entry__ as ge
    ge.build()
    import paper_2604_12672_gb300 as P
    return P


def run(P, pr, fused, dt, eps):
    g = P.Grid(pr, precision="mixed", eps_sf=eps)
    g.set_fused(fused)
    g.load()
    g.step(2, dt)
    out = g.get_state()
    flags = g.test_raw_flags(0)[0] if fused else None
    g.close()
    return out, flags


@pytest.mark.parametrize("recon", ["vanleer", "pph"])
@pytest.mark.parametrize("n", [(32, 64, 38), (32, 76, 32), (32, 77, 32), (40, 64, 32)],
                         ids=["32x64x38-160", "152tiles", "160tiles", "40x64x32-160"])
def test_both_sides_of_one_tile_per_sm(P, n, recon):
    pr = W.stratified_box(*n, amp=5e-2, beta=1e3, mach_heat=3e-2)
    pr.recon = recon
    # a pressure bump: flags around it, none far away
    z, y, x = np.meshgrid(*[(np.arange(k) + 0.5) / k for k in n[::-1]], indexing="ij")
    pr.cons[4] *= 1.0 + 0.3 * np.exp(-((x - 0.1) ** 2 + (y - 0.95) ** 2 + (z - 0.5) ** 2) / 0.01)
    dt = 1e-4
    a, flags = run(P, pr, True, dt, 0.25)
    b, _ = run(P, pr, False, dt, 0.25)
    assert 0 < flags.sum() < flags.size
    for k, v in deviation_l1(pr, a, b).items():
        assert v <= 1e-5, (k, v)
