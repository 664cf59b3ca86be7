"""GPU checks of what the fixed-point contractions (xg_fixed.cuh) owe to each
node, whatever the rest of its tile, its line or the other direction holds: a
constant has no derivative at all."""

import numpy as np
import pytest

from inputs import workloads as W

from helpers import GpuContext

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", range(1, 9))
def test_uniform_fields_have_no_derivative(cuda_device, N):
    """Uniform momentum, rho' and Theta' on periodic levels: every x and y
    derivative is exactly zero, at any spacing and value, in the tendency, the
    linear operator and the hyper-diffusion."""
    import torch
    rng = np.random.RandomState(40 + N)
    for _ in range(12):
        h = 300.0 + 2700.0 * rng.rand(3)
        nel = (3, 2, 2)
        wl = W.box(nel, N, (0.0, 0.0, 0.0), tuple(n * d for n, d in zip(nel, h)), (True, True, False), f=0.0, seed=3)
        wl["S_theta"] = None
        wl["q"] = np.repeat(np.array([1e-3, 7.0, 5.0, 0.0, 0.4]) * rng.uniform(-1.0, 1.0, 5), wl["q"].shape[1]).reshape(5, -1)
        with GpuContext(wl) as g:
            assert not g.rhs()[[0, 1, 2, 4]].any()
            t = torch.from_numpy(wl["q"]).to(cuda_device)
            out = torch.empty_like(t)
            g.xg.xg_linear_operator(g.ctx, t, out)
            assert not out.cpu().numpy()[[0, 1, 2, 4]].any()
            g.xg.xg_set_dynamics(g.ctx, (1e-4, 1e-4, 1e-4), 0.5, 0.0, 0.0)
            g.xg.xg_dynamics_tendency(g.ctx, out)
            assert not out.cpu().numpy().any()
        with GpuContext(wl, precision=2) as g:
            assert not g.rhs()[[0, 4]].any()
