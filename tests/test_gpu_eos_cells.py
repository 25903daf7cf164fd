"""The EOS table's cell polynomials at the places where they can go wrong:
the smallest tables, one-interval-wide directions, states on and beside the
nodes and in the first and last interval, against the oracle's own table and
interpolation.  Bars as in test_batch_inversion_vs_oracle: first derivatives of
f 1e-11, gamma_c (second derivatives, whose node values agree only to ~1e-13 of
|f| + |f_x|) 1e-9."""
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


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("lr, nr, lT, nT", [((5.9, 6.1), 4, (8.9, 9.0), 4), ((5.9, 6.1), 5, (8.0, 9.5), 61),
                                            ((4.0, 8.0), 161, (8.9, 9.0), 4), ((5.0, 7.0), 81, (8.0, 9.5), 61)])
def test_cells_and_edges(P, lr, nr, lT, nT, precision):
    dt, ot = P.EosTable(lr, nr, lT, nT), O.EosTable(lr, nr, lT, nT)
    cfg = O.stellar_cfg(W.STELLAR_A, W.STELLAR_Z, ot)
    # cell positions: just inside the table, on either side of nodes, mid-cell
    def places(n):
        last = n - 1
        return sorted({1e-6, 0.5, 1 - 1e-9, 1 + 1e-9, last / 2 + 0.25, last - 1 - 1e-9, last - 1 + 1e-9, last - 0.5, last - 1e-6})
    Xs = [0.5, 0.5]
    abar, ye = 1.0 / (0.5 / 16.0 + 0.5 / 28.0), 0.5
    rho, T = (a.ravel() for a in np.meshgrid([10 ** (lr[0] + q * (lr[1] - lr[0]) / (nr - 1)) / ye for q in places(nr)],
                                             [10 ** (lT[0] + q * (lT[1] - lT[0]) / (nT - 1)) for q in places(nT)]))
    ref = [O.eos_rt(cfg, r, t, Xs) for r, t in zip(rho, T)]
    e = np.array([r["e"] for r in ref])
    one = np.ones(rho.size)
    inside = [10 ** lT[0] * (1 + 1e-12), 10 ** lT[1] * (1 - 1e-12)]
    out = P.eos(dt, rho, e, abar * one, ye * one, np.clip(T * (1 + 1e-5), *inside), precision=precision)
    inv = [O.eos_invert(cfg, r, q, Xs, t) for r, q, t in zip(rho, e, T)]
    assert np.abs(out["T"] / np.array([r["T"] for r in inv]) - 1).max() <= 1e-11
    for key, tol in (("P", 1e-11), ("gamma_e", 1e-11), ("gamma_c", 1e-9)):
        assert np.abs(out[key] / np.array([r[key] for r in inv]) - 1).max() <= tol, key
    dt.close()


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("nr", [4, 81])
def test_outside_is_refused(P, nr, precision):
    """Densities beside either end of the table, far outside and NaN are
    refused one by one; those just inside converge."""
    lr, lT = (5.0, 7.0), (8.0, 9.5)
    dt, ot = P.EosTable(lr, nr, lT, 61), O.EosTable(lr, nr, lT, 61)
    cfg = O.stellar_cfg(W.STELLAR_A, W.STELLAR_Z, ot)
    ye, T = 0.5, 10 ** 8.7
    last = nr - 1
    place = np.array([1e-9, 0.5, last - 1e-9, -1e-9, -1.0, last + 1e-9, last + 0.5])
    rho = np.append(10 ** (lr[0] + place * (lr[1] - lr[0]) / last) / ye, [1e-200, 1e200, np.nan])
    e = np.full(10, O.eos_rt(cfg, 10 ** 6 / ye, T, [0.5, 0.5])["e"])
    for k in (0, 1, 2):
        e[k] = O.eos_rt(cfg, rho[k], T, [0.5, 0.5])["e"]
    one = np.ones(10)
    out = P.eos(dt, rho, e, one / (0.5 / 16.0 + 0.5 / 28.0), ye * one, T * one * (1 + 1e-5), precision=precision)
    assert (out["iters"][:3] > 0).all() and np.abs(out["T"][:3] / T - 1).max() <= 1e-9
    assert (out["iters"][3:] == -1).all() and np.isnan(out["P"][3:]).all()
    dt.close()
