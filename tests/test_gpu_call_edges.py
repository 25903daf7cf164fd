"""Calls at the edge of what the entry points accept."""
import types

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


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_one_cell_without_active_axes(P, precision):
    """A grid of one cell has no faces, only the gravity source: the momentum
    grows linearly and the energy with its square, which the RK3 step
    integrates exactly (a few roundings in FP64, the FP32 increments' 1e-7 of
    the change in the mixed form)."""
    pr = types.SimpleNamespace(n=(1, 1, 1), lo=(0.0,) * 3, hi=(1.0,) * 3, bc=((0, 0),) * 3, gamma=5 / 3,
                               g=(0.0, 0.0, -1.0), bg=None, heat=None, cfl=0.4, riemann="lhlld", eps_sf=0.2,
                               mach_thr=0.6, nspec=0, eos="ideal")
    cons = np.array([1.0, 0.1, 0.0, 0.0, 2.0]).reshape(5, 1, 1, 1)
    faces = [np.full((1, 1, 2), 0.1), np.full((1, 2, 1), 0.2), np.full((2, 1, 1), 0.3)]
    g = P.Grid(pr, precision=precision)
    g.set_state(cons, *faces)
    g.step(2, 1e-2)
    out = [np.zeros_like(cons)] + [np.zeros_like(f) for f in faces]
    g.get_state_into(*out)
    g.close()
    t = 2e-2
    assert np.abs(out[0].ravel() - [1.0, 0.1, 0.0, -t, 2.0 + 0.5 * t * t]).max() <= (1e-15 if precision == "fp64" else 2e-9)
    for a, b in zip(out[1:], faces):
        assert np.array_equal(a, b)
