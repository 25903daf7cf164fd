"""Faces evaluated in walks along their direction (two or four per thread on
larger grids): FP64 form against the oracle at 1e-11 relative L-infinity where
the face counts leave a remainder, in two and three dimensions, with walls."""
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
    O.set_parallel(True)
    yield P
    O.set_parallel(False)


@pytest.mark.parametrize("pr", [W.orszag_tang(413), W.orszag_tang(790),
                                W.stratified_box(53, 59, 56, amp=3e-2, beta=1e3), W.stratified_box(83, 91, 85, amp=3e-2, beta=1e3)],
                         ids=lambda p: p.name)
def test_walks_match_oracle(P, pr):
    # a flow in every cell, so that no field is rounding noise
    rng = np.random.Generator(np.random.PCG64(9))
    v = 0.05 * rng.uniform(-1.0, 1.0, (3,) + pr.cons.shape[1:])
    pr.cons[4] += 0.5 * pr.cons[0] * (v ** 2).sum(0) + (pr.cons[1:4] * v).sum(0)
    pr.cons[1:4] += pr.cons[0] * v
    g = P.Grid(pr)
    g.load()
    g.step(1)
    st = g.get_state()
    g.close()
    ref, _, _ = O.Oracle(pr).run(1)
    for k in ("bx", "by", "bz"):   # a field that starts at zero: against the vector's scale
        scale = max(np.abs(ref[q]).max() for q in ("bx", "by", "bz"))
        assert np.abs(st[k] - ref[k]).max() <= 1e-11 * scale, k
    for q in range(5):
        scale = np.abs(ref["cons"][1:4]).max() if 1 <= q <= 3 else np.abs(ref["cons"][q]).max()
        assert np.abs(st["cons"][q] - ref["cons"][q]).max() <= 1e-11 * scale, q
