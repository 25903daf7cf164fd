"""The state layout kernel: what set_state loads, get_state returns bit for bit,
for odd and even x extents (one and two doubles per unit), one to three active
dimensions, mass fractions, fields of fewer and more elements than a block, and
device arrays that do not start on 16 bytes."""
import types

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    import torch
    assert torch.cuda.is_available()
    import __graft_entry__ as ge
    ge.build()
    import paper_2604_12672_gb300 as P
    return P


@pytest.mark.parametrize("where", ["host", "device", "device+8"])
@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("n, nspec", [((4, 1, 1), 0), ((37, 1, 1), 2), ((64, 50, 1), 0), ((33, 7, 1), 0),
                                      ((16, 12, 9), 0), ((17, 5, 6), 4), ((130, 31, 33), 1)])
def test_round_trip(P, n, nspec, precision, where):
    import torch
    pr = types.SimpleNamespace(n=n, lo=(0.0,) * 3, hi=(1.0,) * 3, bc=((0, 0),) * 3, gamma=5 / 3, g=(0.0,) * 3, bg=None,
                               heat=None, cfl=0.4, riemann="lhlld", eps_sf=0.2, mach_thr=0.6, nspec=nspec, eos="ideal")
    rng = np.random.default_rng(5)
    nx, ny, nz = n
    shapes = [(5 + nspec, nz, ny, nx), (nz, ny, nx + 1), (nz, ny + 1, nx), (nz + 1, ny, nx)]
    src = [rng.uniform(1.0, 2.0, s) for s in shapes]
    g = P.Grid(pr, precision=precision)
    if where == "host":
        out = [np.zeros(s) for s in shapes]
        g.set_state(*src)
        g.get_state_into(*out)
        got = out
    else:
        off = 1 if where == "device+8" else 0   # doubles
        def dev(a):
            buf = torch.zeros(a.size + off, dtype=torch.float64, device="cuda")
            return buf[off:].reshape(a.shape)
        a, out = [dev(s) for s in src], [dev(s) for s in src]
        for t, s in zip(a, src):
            t.copy_(torch.from_numpy(s))
        g.set_state(*a)
        g.get_state_into(*out)
        torch.cuda.synchronize()
        got = [t.cpu().numpy() for t in out]
    g.close()
    for x, y in zip(got, src):
        assert np.array_equal(x, y)
