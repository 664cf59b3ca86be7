"""GPU checks of the fixed-point line contractions (xg_fixed.cuh) behind the
linear operator and the weak Laplacian: every order, tiles that are full,
ragged and single, every kind of end; values of widely different size in one
tile; and an infinity or NaN, which must reach no further than the FP64 chains
would carry it."""

import numpy as np
import pytest

from inputs import workloads as W
from oracle import dynamics as Y, euler as E, imex as X

from helpers import GpuContext, oracle_of, rel_l2_per_var

pytestmark = pytest.mark.gpu

MESHES = [((1, 1, 1), (False, False, False)), ((1, 2, 1), (True, True, True)), ((9, 3, 2), (False, True, False)),
          ((5, 11, 3), (True, False, True)), ("tile", (False, True, False)), ("tile", (False, False, False))]


def _case(nel, N, per):
    if nel == "tile":   # exactly one tile along x, two and a bit along y
        nel = (32 // N, 2 * (32 // N) + 1, 1)
    elif N <= 2:   # more than one tile of 32 / N elements
        nel = (nel[0] * 4, nel[1] * 4, nel[2])
    return W.box(nel, N, (0.0, 0.0, 0.0), (1000.0 * nel[0], 700.0 * nel[1], 400.0 * nel[2]), per, seed=17)


def _operator(g, v, dev):
    import torch
    t = torch.from_numpy(v).to(dev)
    out = torch.empty_like(t)
    g.xg.xg_linear_operator(g.ctx, t, out)
    return out.cpu().numpy()


@pytest.mark.parametrize("N", range(1, 9))
@pytest.mark.parametrize("nel,per", MESHES)
def test_operators_match_oracle(cuda_device, nel, per, N):
    import torch
    wl = _case(nel, N, per)
    m, phys, base = oracle_of(wl)
    with GpuContext(wl) as g:
        L = _operator(g, wl["q"], cuda_device)
        g.xg.xg_set_dynamics(g.ctx, (1e-4, 1e-4, 1e-4), 0.5, 0.0, 0.0)
        H = torch.empty((5, g.np), dtype=torch.float64, device=cuda_device)
        g.xg.xg_dynamics_tendency(g.ctx, H)
        H = H.cpu().numpy()
    assert np.all(rel_l2_per_var(L, X.linear_operator(m, wl["q"], base, phys)) <= 1e-12)
    tau = Y.viscosity_tensor(m, (1e-4, 1e-4, 1e-4), 0.5)
    assert np.all(rel_l2_per_var(H, Y.hyperdiffusion(m, wl["q"], tau)) <= 1e-12)


def test_wide_range_of_values(cuda_device):
    """A field that falls by 2^-40 within a tile: the error stays at FP64's
    rounding of the tile's largest values."""
    wl = _case((9, 3, 2), 4, (False, True, False))
    m, phys, base = oracle_of(wl)
    v = wl["q"] * np.exp2(-40.0 * np.linspace(0.0, 1.0, m.n[0]))[np.arange(m.Np) % m.n[0]]
    with GpuContext(wl) as g:
        L = _operator(g, v, cuda_device)
    ref = X.linear_operator(m, v, base, phys)
    assert np.all(rel_l2_per_var(L, ref) <= 1e-12)


@pytest.mark.parametrize("bad", [np.nan, np.inf])
@pytest.mark.parametrize("var", [1, 2, 3, 4])
def test_nonfinite_reaches_its_own_lines_only(cuda_device, var, bad):
    """(The oracle's general metric terms multiply the other directions by
    zero, which carries a NaN across its whole element, so the reach is
    written out here: the node's element segment along the direction that
    each equation differentiates the variable in.)"""
    wl = _case((9, 3, 2), 4, (False, True, False))
    m, phys, base = oracle_of(wl)
    at = (m.n[0] // 2 + 1, 5, 3)                    # inside an element in every direction
    v = wl["q"].copy()
    v[var, at[0] + m.n[0] * (at[1] + m.n[1] * at[2])] = bad
    clean = X.linear_operator(m, wl["q"], base, phys)
    with GpuContext(wl) as g:
        L = _operator(g, v, cuda_device)
    fine = np.ones((5,) + tuple(m.n[::-1]), dtype=bool)
    reach = {1: [(0, 0), (4, 0)], 2: [(0, 1), (4, 1)], 3: [(0, 2), (4, 2)], 4: [(1, 0), (2, 1), (3, 2)]}[var]
    for eq, d in reach:
        sel = [at[2], at[1], at[0]]
        e = at[d] // 4
        sel[2 - d] = slice(4 * e, 4 * e + 5)
        fine[(eq,) + tuple(sel)] = False
    if var == 4:
        fine[3, 0] = True                           # the wall's zero
    fine = fine.reshape(5, -1)
    assert np.array_equal(np.isfinite(L), fine)
    assert np.allclose(L[fine], clean[fine], rtol=1e-9, atol=1e-12 * np.abs(clean).max())
