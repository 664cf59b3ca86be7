"""GPU check of the centroids' sums (xg_ri_velocity), whose terms have both
signs, against extended precision."""

import numpy as np
import pytest

from inputs import grid, workloads as W

from helpers import GpuContext

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("seed", [1, 2, 3])
def test_centroids_against_extended_precision(cuda_device, seed):
    """400 x 400 columns.  A row is a warp's: its lanes add some 13 terms and the
    lanes are added in five steps, so a warp's sum of s x is rounded at about
    sqrt(18) 2^-54 of what it holds, and the 400 warps' errors, independent, at
    sqrt(18 / 400) 2^-54 of all of it: 0.1 x 2^-53 of the half width, whose
    largest of 10 is below 2^-55 of it.  The warps' sums are added with their
    remainders; the two totals and their quotient are rounded once each."""
    nel = (100, 100, 1)
    wl = W.tc(nel=nel, state="random", seed=seed)
    n = [4 * nel[0], 4 * nel[1], 4 * nel[2] + 1]
    with GpuContext(wl) as g:
        _, cent, _ = g.xg.xg_ri_velocity(g.ctx, 5)
    _, _, _, ax = grid.node_coords(wl["nel"], wl["N"], wl["lo"], wl["hi"], wl["periodic"])
    q = wl["q"].astype(np.longdouble).reshape(5, n[2], n[1], n[0])
    rho = wl["rho0"].astype(np.longdouble)[:, None, None] + q[0]
    s = np.sqrt(q[1] ** 2 + q[2] ** 2 + q[3] ** 2) / rho
    x, y = (a.astype(np.longdouble) for a in ax[:2])
    ref = np.stack([(s * x).sum(axis=(1, 2)), (s * y[:, None]).sum(axis=(1, 2))], axis=1) / s.sum(axis=(1, 2))[:, None]
    err = np.abs(np.asarray(cent).reshape(ref.shape) - ref)
    tol = 2.0 ** -55 * max(abs(x[0]), abs(y[0])) + 3 * 2.0 ** -53 * np.abs(ref)
    assert np.all(err <= tol), float((err / tol).max())
