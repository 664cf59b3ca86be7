"""GPU checks of the mixed form's two sets of x and y kernels: which one a box
takes, and the line kernels on slabs against their domain, bit for bit."""

import numpy as np
import pytest

from inputs import workloads as W
from paper_2504_08157_gb300 import partition as P

from helpers import GpuContext
from test_gpu_partition import _slabs as slabs_of

pytestmark = pytest.mark.gpu

DF64 = 2


def _box(nel, N, per, seed=37):
    return W.box(nel, N, (0.0, 0.0, 0.0), (1000.0 * nel[0], 800.0 * nel[1], 500.0 * nel[2]), per, f=1.0e-4, seed=seed)


def _takes_lines(g):
    """Whether a right-hand side launched the y line kernel (timing slot 1)."""
    import torch
    g.xg.xg_profile(g.ctx, True)
    g.rhs()
    torch.cuda.synchronize()
    _, launches = g.xg.xg_kernel_times(g.ctx)
    g.xg.xg_profile(g.ctx, False)
    return launches[1] > 0


# the longest x line of each order that the tiles take (0: none)
LONGEST = {1: 0, 2: 64, 3: 48, 4: 96, 5: 90}


@pytest.mark.parametrize("ny,nz", [(1, 1), (2, 7), (60, 1)])
@pytest.mark.parametrize("N", range(1, 6))
def test_path_by_the_length_of_x_lines_alone(cuda_device, N, ny, nz):
    """Beyond the crossover a box takes the lines however few levels it has: the
    tiles cost more there once n_y fills the chip, and a slab must take the path
    of its domain whatever its n_y."""
    most = LONGEST[N] // N
    for nx, lines in ((most, False), (most + 1, True), (max(most + 1, 200 // N), True)):
        if nx == 0:
            continue
        with GpuContext(_box((nx, ny, nz), N, (True, True, False)), precision=DF64) as g:
            assert _takes_lines(g) == lines, nx


@pytest.mark.parametrize("per_y", [True, False])
@pytest.mark.parametrize("parts", [2, 3])
@pytest.mark.parametrize("N,nx", [(1, 2060), (2, 700), (3, 350), (4, 210), (5, 140)])
def test_slabs_on_lines_equal_the_domain(cuda_device, N, nx, parts, per_y):
    import torch
    wl = _box((nx, 7, 1), N, (True, per_y, False))
    with GpuContext(wl, precision=DF64) as g:
        assert _takes_lines(g)
        r_ref = g.rhs()
        g.step(2)
        q_ref = g.state()
    ctxs = slabs_of(wl, parts, DF64)
    try:
        slabs = [c.s for c in ctxs]
        outs = [torch.empty((5, c.np), dtype=torch.float64, device=cuda_device) for c in ctxs]
        P.rhs(ctxs, outs)
        torch.cuda.synchronize()
        for o, s in zip(outs, slabs):
            assert np.array_equal(o.cpu().numpy(), P.scatter(r_ref, s))
        P.step(ctxs, wl["dt"], 2)
        for c, s in zip(ctxs, slabs):
            assert np.array_equal(c.state().cpu().numpy(), P.scatter(q_ref, s))
    finally:
        for c in ctxs:
            c.close()
