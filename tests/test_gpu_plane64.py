"""GPU checks of the FP64-accurate x-y tile kernel and the z passes behind it
(xg_plane64.cuh): every order on meshes that fill one tile exactly, spill over
it in x and in y, or close on themselves, with every kind of end; and an
infinity or NaN, which must reach its own lines only."""

import numpy as np
import pytest

from inputs import workloads as W
from oracle import euler as E

from helpers import GpuContext, oracle_of, rel_l2_per_var

pytestmark = pytest.mark.gpu

ROWS = {1: 9, 2: 4, 3: 3, 4: 2, 5: 1, 6: 1, 7: 1, 8: 1}   # element rows of a tile


def _mesh(N, kind):
    ex, ey = 32 // N, ROWS[N]
    return {"exact": (ex, ey, 1), "spill": (ex + 1, 2 * ey + 1, 2), "one": (1, 1, 2)}[kind]


@pytest.mark.parametrize("prec", [0, 2], ids=["fp64", "df64"])
@pytest.mark.parametrize("per", [(False, False, False), (True, True, False), (False, True, True), (True, False, False)])
@pytest.mark.parametrize("kind", ["exact", "spill", "one"])
@pytest.mark.parametrize("N", range(1, 9))
def test_rhs_matches_oracle(cuda_device, N, kind, per, prec):
    if kind == "one" and prec == 2:
        pytest.skip("a momentum part that vanishes on one periodic element leaves 48-bit rounding of its fluxes")
    nel = _mesh(N, kind)
    wl = W.box(nel, N, (0.0, 0.0, 0.0), (1000.0 * nel[0], 800.0 * nel[1], 500.0 * nel[2]), per, f=1.0e-4, seed=29)
    m, phys, base = oracle_of(wl)
    ref = E.rhs(m, wl["q"], base, wl["S_theta"], phys)
    with GpuContext(wl, precision=prec) as g:
        got = g.rhs()
    assert np.all(rel_l2_per_var(got, ref) <= 1e-12)


@pytest.mark.parametrize("prec", [0, 2], ids=["fp64", "df64"])
@pytest.mark.parametrize("bad", [np.nan, np.inf])
@pytest.mark.parametrize("at", [(35, 9, 5), (32, 8, 4), (3, 3, 0)])
def test_nonfinite_reaches_its_own_lines_only(cuda_device, at, bad, prec):
    """A non-finite rho u changes every equation's x part and the momentum's
    and Theta's y and z parts, on the element segments that hold the node."""
    wl = W.box((9, 5, 2), 4, (0.0, 0.0, 0.0), (9000.0, 5000.0, 1000.0), (False, True, False), seed=31)
    m, phys, base = oracle_of(wl)
    clean = E.rhs(m, wl["q"], base, wl["S_theta"], phys)
    q = wl["q"].copy()
    q[1, at[0] + m.n[0] * (at[1] + m.n[1] * at[2])] = bad
    bad_wl = dict(wl, q=q)
    with GpuContext(bad_wl, precision=prec) as g:
        got = g.rhs()
    fine = np.ones(tuple(m.n[::-1]), dtype=bool)
    for d in range(3):
        sel = [at[2], at[1], at[0]]
        n, per = m.n[d], wl["periodic"][d]
        segs = {at[d] // 4} | ({at[d] // 4 - 1} if at[d] % 4 == 0 else set())
        nodes = set()
        for e in segs:
            if per or 0 <= e < wl["nel"][d]:
                nodes |= {(4 * (e % wl["nel"][d]) + a) % n for a in range(5)}
        sel[2 - d] = sorted(nodes)
        fine[tuple(sel)] = False
    fine = np.broadcast_to(fine.reshape(-1), got.shape)
    assert np.all(np.isfinite(got[fine]))
    assert np.allclose(got[fine], clean[fine], rtol=1e-9, atol=1e-9 * np.abs(clean).max())
    assert not np.isfinite(got[1, at[0] + m.n[0] * (at[1] + m.n[1] * at[2])]) or at[0] in (0, m.n[0] - 1)
