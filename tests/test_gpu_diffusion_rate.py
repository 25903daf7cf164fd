"""The stage count of the diffusion step: the parabolic rate's maximum is found
from integer keys of the cells' products, so fields whose maximum sits in one
cell, in equal cells, or beside products within an FP32 rounding of it must give
the rate of the FP64 product of every cell."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    import __graft_entry__ as ge
    ge.build()
    import paper_2604_12672_gb300 as P
    return P


@pytest.mark.parametrize("form", ["fp64", "mixed"])
@pytest.mark.parametrize("nT, nR", [(0, 0), (3, 1), (4, 2)])
@pytest.mark.parametrize("field", ["one cell", "equal", "close"])
def test_stage_count_of_the_largest_rate(P, form, nT, nR, field):
    n = (17, 9, 12)
    pr = W.stratified_box(*n, amp=0.0, beta=1e3, mach_heat=0.0)
    r = np.random.default_rng(3)
    rho = np.ones(n[::-1])
    e = np.ones(n[::-1])
    if field == "one cell":
        rho, e = 1.0 + 0.2 * r.random(rho.shape), 1.0 + 0.2 * r.random(e.shape)
        e[7, 4, 11] = 1.5
    elif field == "close":   # products a few FP64 roundings apart
        e = 1.0 + 1e-13 * r.random(e.shape)
    for f in (pr.bx, pr.by, pr.bz):
        f[...] = 0.0
    pr.cons[...] = 0.0
    pr.cons[0], pr.cons[4] = rho, rho * e
    D = 1e-3 * e ** nT / rho ** (nR + 1)
    rate = D.max() * sum(1.0 / d ** 2 for d in pr.dx())
    # the count steps from 9 to 10 at dt / dt_p = (9^2 + 9 - 2) / 4
    for s, eps, want in ((9, -1e-6, 9), (9, 1e-6, 10)):
        g = P.Grid(pr, precision=form)
        g.load()
        got = g.diffuse((s * s + s - 2) / 4 * (1 + eps) * 0.5 / rate, k0=1e-3, nT=nT, nR=nR, cv=1.0)
        g.close()
        assert got == want, (got, want)
