"""The tile kernel's form for grids of at most one tile per SM (one face per
thread, the raw flags dilated in the tile): well below that line, exactly on
it with whole and partial tiles, and one tile above it, with part of the cells
flagged -- against the per-direction kernels with their own dilation passes.  The
mixed form's bar, 1e-5 relative L1 of the deviations: a tile that missed its
neighbours' flags would take another solver on the faces beside them."""
import numpy as np
import pytest

import workloads as W
from test_gpu_mixed import deviation_l1
from test_gpu_small_tiles import P, run  # noqa: F401 (fixture)

pytestmark = pytest.mark.gpu


def threshold(pr):
    """A flattening threshold that about a fifth of the cells exceed, in the
    middle of the widest gap between their indicators (sum over the axes of
    |P_(i+1) - P_(i-1)| over P), so that rounding decides no cell."""
    c = pr.cons
    b2 = sum((0.5 * (f.take(range(1, f.shape[ax]), ax) + f.take(range(f.shape[ax] - 1), ax))) ** 2
             for f, ax in ((pr.bx, 2), (pr.by, 1), (pr.bz, 0)))
    p = (pr.gamma - 1) * (c[4] - 0.5 * (c[1:4] ** 2).sum(0) / c[0] - 0.5 * b2)
    s = sum(np.abs(np.roll(p, -1, ax) - np.roll(p, 1, ax)) for ax in range(3))[1:-1] / p[1:-1]
    v = np.sort(s.ravel())
    v = v[int(0.75 * v.size): int(0.85 * v.size) + 2]
    k = np.argmax(np.diff(v) / v[1:])
    return 0.5 * (v[k] + v[k + 1])


@pytest.mark.parametrize("recon", ["vanleer", "pph"])
@pytest.mark.parametrize("n, tiles", [((8, 16, 12), 4), ((20, 12, 37), 30), ((32, 32, 48), 96), ((16, 32, 152), 152),
                                      ((15, 31, 149), 152), ((24, 24, 136), 153)])
def test_forms_agree(P, n, tiles, recon):  # noqa: F811
    import torch
    assert np.prod([(k + 7) // 8 for k in n]) == tiles
    assert torch.cuda.get_device_properties(0).multi_processor_count == 152   # the line the sizes straddle
    pr = W.stratified_box(*n, amp=5e-2, beta=1e3, mach_heat=3e-2)
    pr.recon = recon
    # a pressure bump across a periodic side
    z, y, x = np.meshgrid(*[(np.arange(k) + 0.5) / k for k in n[::-1]], indexing="ij")
    pr.cons[4] *= 1.0 + 0.3 * np.exp(-((x - 0.1) ** 2 + (y - 0.95) ** 2 + (z - 0.5) ** 2) / 0.01)
    eps = threshold(pr)
    a, flags = run(P, pr, True, 1e-4, eps)
    b, _ = run(P, pr, False, 1e-4, eps)
    c, _ = run(P, pr, False, 1e-4, 1e3)   # nothing flagged: what the flags are worth
    assert deviation_l1(pr, c, b)["m"] > 1e-3
    assert 0 < flags.sum() < flags.size
    for k, v in deviation_l1(pr, a, b).items():
        assert v <= 1e-5, (k, v)
