"""The tile kernel away from and at the boundaries (tiles that touch none skip
the tests for faces outside the domain and at walls), with no cell flagged (no
flags staged) and some, on sizes that leave partial tiles along every axis:
against the per-direction kernels, the mixed form's bar, 1e-5 relative L1 of
the deviations."""
import numpy as np
import pytest

import workloads as W
from test_gpu_mixed import deviation_l1
from test_gpu_small_tiles import P, run  # noqa: F401 (fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("recon", ["vanleer", "pph"])
@pytest.mark.parametrize("flagged", [False, True])
@pytest.mark.parametrize("n", [(40, 67, 61), (25, 81, 47)], ids=["40x67x61", "25x81x47"])
def test_inner_and_boundary_tiles(P, n, flagged, recon):  # noqa: F811
    pr = W.stratified_box(*n, amp=5e-2, beta=1e3, mach_heat=3e-2)
    pr.recon = recon
    if flagged:   # a pressure bump across an inner tile corner and a side
        z, y, x = np.meshgrid(*[(np.arange(k) + 0.5) / k for k in n[::-1]], indexing="ij")
        pr.cons[4] *= 1.0 + 0.3 * np.exp(-((x - 0.4) ** 2 + (y - 0.95) ** 2 + (z - 0.5) ** 2) / 0.01)
    eps = 0.25 if flagged else 1e3   # a threshold no cell reaches
    a, flags = run(P, pr, True, 1e-4, eps)
    b, _ = run(P, pr, False, 1e-4, eps)
    assert (flags.sum() > 0) == flagged and flags.sum() < flags.size
    for k, v in deviation_l1(pr, a, b).items():
        assert v <= 1e-5, (k, v)
