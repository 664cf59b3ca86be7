"""GPU checks of the mixed form's two sets of x and y kernels: which one a box
takes, and the line kernels on the boxes that only long x lines reach -- every
order and kind of end, more segments than a block has threads, y tiles that close
on themselves, partitions, infinities and NaN."""

import numpy as np
import pytest

from inputs import workloads as W
from paper_2504_08157_gb300 import partition as P

from helpers import GpuContext, oracle_of
from test_gpu_fixed_limits import TOL, Lines
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
LONGEST = {1: 0, 2: 64, 3: 60, 4: 96, 5: 90}


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


# A row, the sums over directions and the result of the double-float momentum:
# sixteen roundings of 2^-46 (rho' and Theta' keep the FP64 allowance).
TOL_DF = 16 * 2.0 ** -46


def _check_rhs(wl, lines):
    ref, (_, phys, _) = Lines(wl), oracle_of(wl)
    L, top = ref.rhs(wl["q"], phys)
    with GpuContext(wl, precision=DF64) as g:
        assert _takes_lines(g) == lines
        got = g.rhs().reshape((5,) + L[0].shape)
    for v in range(5):
        tol = TOL if v in (0, 4) else TOL_DF
        worst = float((np.abs(got[v] - L[v]) / (tol * top[v] + np.longdouble(1e-300))).max())
        assert worst <= 1.0, (v, worst)


ENDS = [(False, False, False), (True, True, False), (False, True, True), (True, False, False)]


@pytest.mark.parametrize("per", ENDS)
@pytest.mark.parametrize("N,nel", [(1, (20, 7, 1)), (1, (140, 1, 1)), (2, (33, 9, 1)), (2, (133, 1, 1)), (3, (21, 7, 1)),
                                   (3, (130, 1, 1)), (4, (25, 1, 1)), (4, (25, 5, 2)), (4, (130, 2, 1)), (5, (19, 1, 1)),
                                   (5, (19, 3, 1))])
def test_line_kernels_match_extended_precision(cuda_device, N, nel, per):
    wl = _box(nel, N, per)
    wl["S_theta"] = None
    _check_rhs(wl, True)


@pytest.mark.parametrize("per", ENDS + [(True, True, True)])
@pytest.mark.parametrize("N", range(1, 9))
def test_single_elements_in_the_tiles(cuda_device, N, per):
    """One element along x and y: a part of the momentum that vanishes on a
    periodic element leaves the rounding of its fluxes, which is what the
    allowance is measured by."""
    wl = _box((1, 1, 2), N, per)
    wl["S_theta"] = None
    _check_rhs(wl, N == 1)


@pytest.mark.parametrize("bad", [np.nan, np.inf])
@pytest.mark.parametrize("at", [(50, 9, 5), (48, 8, 4), (3, 3, 0), (99, 0, 2)])
def test_nonfinite_reaches_its_own_lines_only(cuda_device, at, bad):
    """A non-finite rho u changes every equation's x part and the momentum's
    and Theta's y and z parts, on the element segments that hold the node."""
    wl = _box((25, 5, 2), 4, (True, True, False), seed=31)
    n, nel, per = (100, 20, 9), wl["nel"], wl["periodic"]
    with GpuContext(wl, precision=DF64) as g:
        assert _takes_lines(g)
        clean = g.rhs()
        q = wl["q"].copy()
        node = at[0] + n[0] * (at[1] + n[1] * at[2])
        q[1, node] = bad
        g.set_state(q)
        got = g.rhs()
    fine = np.ones(n[::-1], dtype=bool)
    for d in range(3):
        nodes = set()
        for e in {at[d] // 4} | ({at[d] // 4 - 1} if at[d] % 4 == 0 else set()):
            if per[d] or 0 <= e < nel[d]:
                nodes |= {(4 * (e % nel[d]) + a) % n[d] for a in range(5)}
        sel = [at[2], at[1], at[0]]
        sel[2 - d] = sorted(nodes)
        fine[tuple(sel)] = False
    fine = np.broadcast_to(fine.reshape(-1), got.shape)
    assert np.array_equal(got[fine], clean[fine])
    assert not np.isfinite(got[1, node])


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


@pytest.mark.parametrize("N", [1, 2, 3, 4])
def test_tile_height_leaves_the_bits_alone(cuda_device, N):
    """A context of few levels cuts its tiles to fewer element rows than the
    allocation-free call, which takes the full height."""
    import torch
    wl = _box((3, 19, 1), N, (False, True, False))
    with GpuContext(wl) as g:
        a = g.rhs()
        t = lambda x: torch.from_numpy(np.ascontiguousarray(x)).to(cuda_device)  # noqa: E731
        ph = wl["phys"]
        desc = g.xg.mesh_desc(wl["nel"], N, wl["lo"], wl["hi"], wl["periodic"], f=ph["f"], g=ph["g"], R=ph["R"],
                              cp=ph["cp"], cv=ph["cv"], p_a=ph["p_a"])
        out = torch.empty((5, g.np), dtype=torch.float64, device=cuda_device)
        g.xg.xg_rhs_noalloc(desc, t(wl["q"]), t(wl["rho0"]), t(wl["Theta0"]), t(wl["S_theta"]), out)
        torch.cuda.synchronize()
    assert np.array_equal(a, out.cpu().numpy())
