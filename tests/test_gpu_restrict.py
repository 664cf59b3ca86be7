"""GPU checks of the restriction's passes (k_interp_z, k_interp_y, k_interp_x):
boxes refined by two (half of the coarse nodes fall on fine ones), by no whole
factor and to another order, single elements that close on themselves, enough
planes for several chunks, a result written over its source, and a NaN, which
reaches the coarse nodes of the fine element that holds it and no others."""

import numpy as np
import pytest

from inputs import workloads as W
from oracle import closure as OC

from helpers import GpuContext

pytestmark = pytest.mark.gpu


def _box(nel, N, per):
    return W.box(nel, N, (0.0, 0.0, 0.0), (6000.0, 4000.0, 3000.0), per, seed=41)


def _axes(wl):
    return [(wl["nel"][d], wl["N"], wl["lo"][d], wl["hi"][d], wl["periodic"][d]) for d in range(3)]


CASES = [((8, 6, 4), 4, (4, 3, 2), 4, (False, True, False)), ((5, 7, 3), 3, (3, 2, 2), 5, (True, False, False)),
         ((1, 1, 1), 4, (1, 1, 1), 4, (True, True, False)), ((2, 3, 4), 8, (3, 3, 3), 1, (False, False, True)),
         ((40, 36, 6), 4, (20, 18, 6), 4, (True, True, False))]


@pytest.mark.parametrize("over", [False, True])
@pytest.mark.parametrize("nf,Nf,nc,Nc,per", CASES)
def test_restriction_matches_oracle(cuda_device, nf, Nf, nc, Nc, per, over):
    import torch
    fine, coarse = _box(nf, Nf, per), _box(nc, Nc, per)
    q = fine["q"]
    ref = OC.restrict(_axes(fine), _axes(coarse), q)
    with GpuContext(fine, precision=1) as gf, GpuContext(coarse, precision=1) as gc:
        n = max(q.size, ref.size)
        src = torch.zeros(n, dtype=torch.float64, device=cuda_device)
        src[:q.size] = torch.from_numpy(q.reshape(-1)).to(cuda_device)
        dst = src[:ref.size] if over else torch.empty(ref.size, dtype=torch.float64, device=cuda_device)
        gf.xg.xg_restrict(gf.ctx, gc.ctx, src[:q.size].view(q.shape), dst.view(ref.shape))
        got = dst.cpu().numpy().reshape(ref.shape)
    assert np.all(np.abs(got - ref) <= 1e-13 * np.abs(q).max(axis=1, keepdims=True))


def test_nan_reaches_its_fine_elements(cuda_device):
    import torch
    nf, nc, per = (8, 6, 4), (4, 3, 2), (False, True, False)
    fine, coarse = _box(nf, 4, per), _box(nc, 4, per)
    q = fine["q"].copy()
    n = [4 * nf[0] + 1, 4 * nf[1], 4 * nf[2] + 1]
    q[2, 9 + n[0] * (14 + n[1] * 6)] = np.nan          # inside fine element (2, 3, 1)
    with GpuContext(fine, precision=1) as gf, GpuContext(coarse, precision=1) as gc:
        dst = torch.empty((5, gc.np), dtype=torch.float64, device=cuda_device)
        gf.xg.xg_restrict(gf.ctx, gc.ctx, torch.from_numpy(q).to(cuda_device), dst)
        got = np.isnan(dst.cpu().numpy()).reshape(5, 9, 12, 17)
    # the coarse nodes inside that element, and those on its faces only where
    # the face's value is taken from it
    sure, may = np.zeros_like(got), np.zeros_like(got)
    sure[2, 3:4, 7:8, 4:6] = True
    may[2, 2:4, 6:8, 4:7] = True
    assert np.all(got[sure]) and not np.any(got[~may])
