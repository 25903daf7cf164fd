"""Calls at the edge of what the entry points accept."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    import __graft_entry__ as ge
    ge.build()
    import paper_2604_12672_gb300 as P
    return P


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_eos_without_ions(P, precision):
    """An infinite mean mass number (no ions) is the limit of large ones: at
    1e300 the ions' terms are below 1e-250 of every sum, so both give the same
    bits."""
    t = P.EosTable((4.0, 8.0), 81, (8.0, 9.5), 61)
    rho, T = np.array([1e5, 3e5, 1e6, 2e6]), np.array([3e8, 4e8, 5e8, 1e9])
    e, one = np.full(4, 5e17), np.ones(4)
    a = P.eos(t, rho, e, np.inf * one, 0.5 * one, T, precision=precision)
    b = P.eos(t, rho, e, 1e300 * one, 0.5 * one, T, precision=precision)
    t.close()
    assert (b["iters"][:2] > 0).all()
    for k in a:
        assert np.array_equal(a[k], b[k], equal_nan=True), k
