"""GPU checks of the intensity diagnostics' kernels (xg_ri_velocity,
xg_diagnostics) against the oracle, at rows shorter and longer than a warp,
strips narrower than the node spacing and a single strip."""

import numpy as np
import pytest

from inputs import workloads as W
from oracle import dynamics as Y, euler as E

from helpers import GpuContext, oracle_of

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [0, 1, 2], ids=["fp64", "fp32", "df64"])
@pytest.mark.parametrize("nel,nstrips", [((1, 1, 1), 3), ((7, 9, 2), 1), ((9, 5, 1), 1024), ((17, 8, 2), 20)])
def test_ri_velocity_and_sums(cuda_device, nel, nstrips, prec):
    wl = W.box(nel, 4, (0.0, 0.0, 0.0), tuple(1000.0 * n for n in nel), (True, False, False), seed=5)
    with GpuContext(wl, precision=prec) as g:
        u, cent, means = g.xg.xg_ri_velocity(g.ctx, nstrips)
        sums = np.array(g.xg.xg_diagnostics(g.ctx))
        q = g.state()
    m, _, _ = oracle_of(wl)
    ru, rcent, rmeans = Y.ri_velocity(m, q, wl["rho0"], nstrips=nstrips)
    # sums of n ~ 1e4 positive terms of a few roundings each, in another order
    assert np.allclose(cent, rcent, rtol=1e-12, atol=1e-12 * max(wl["hi"][:2]))
    # the oracle's I - e_r e_r cancels: a few roundings of |u| stay in u_theta
    umax = np.abs(q[1:3]).max() / wl["rho0"].min()
    assert np.allclose(means, rmeans, rtol=1e-12, atol=16 * 2.0 ** -52 * umax)
    assert abs(u - ru) <= 1e-12 * ru
    M = E.mass(m)
    assert np.all(np.abs(sums - (M * q).sum(axis=1)) <= 1e-13 * (M * np.abs(q)).sum(axis=1))


def test_ri_velocity_at_rest(cuda_device):
    wl = W.box((3, 3, 1), 4, (0.0, 0.0, 0.0), (3000.0, 3000.0, 1000.0), (True, True, False), seed=5)
    wl["q"] = np.zeros_like(wl["q"])
    with GpuContext(wl) as g:
        u, cent, means = g.xg.xg_ri_velocity(g.ctx, 7)
    assert u == 0.0 and not means.any() and np.all(cent == 1500.0)
