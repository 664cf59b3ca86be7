"""GPU checks that boxes of few columns, lines or levels keep their results and
cost about what their nodes cost elsewhere: kernels that work on tiles of a level,
on rows or on columns must not leave most of the chip idle on them."""

import pytest

from inputs import workloads as W
from oracle import euler as E

from helpers import GpuContext, oracle_of
from test_gpu_fixed_limits import _check as check_nodes

pytestmark = pytest.mark.gpu

# order 4, about 50,000 nodes each, and a box of as many that fills the tiles
THIN = {"column": (1, 1, 780), "pencil": (1, 3100, 1), "sheet": (1, 60, 52)}
FULL = (16, 16, 3)


def _time(call):
    """Device microseconds of a call, the least of several."""
    import torch
    best = float("inf")
    for _ in range(6):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        torch.cuda.synchronize()
        a.record()
        for _ in range(10):
            call()
        b.record()
        torch.cuda.synchronize()
        best = min(best, a.elapsed_time(b) * 100.0)
    return best


def _box(nel, N=4, per=(False, True, False)):
    return W.box(nel, N, (0.0, 0.0, 0.0), (1000.0 * nel[0], 1000.0 * nel[1], 10.0e3), per, seed=13)


def _operators(g, q):
    import torch
    g.xg.xg_set_dynamics(g.ctx, (1e-4, 1e-4, 1e-4), 0.5, 0.0, 0.0)
    out = torch.empty_like(q)
    return {"linear": lambda: g.xg.xg_linear_operator(g.ctx, q, out),
            "hyper": lambda: g.xg.xg_dynamics_tendency(g.ctx, out)}, out


@pytest.mark.parametrize("shape", sorted(THIN))
def test_operators_cost_on_thin_boxes(cuda_device, shape):
    """A node of a thin box costs at most four times one of a full tile."""
    import torch
    t = {}
    for nel in (THIN[shape], FULL):
        wl = _box(nel)
        with GpuContext(wl) as g:
            q = torch.from_numpy(wl["q"]).to(cuda_device)
            calls, _ = _operators(g, q)
            t[nel] = {k: _time(c) / g.np for k, c in calls.items()}
    ratio = {k: t[THIN[shape]][k] / t[FULL][k] for k in t[FULL]}
    assert max(ratio.values()) <= 4.0, ratio


@pytest.mark.parametrize("nel,per", [((1, 1, 9), (False, False, False)), ((1, 7, 3), (False, True, False)),
                                     ((7, 1, 3), (True, False, False)), ((4, 3, 70), (True, True, False))])
@pytest.mark.parametrize("N", [1, 2, 4, 5, 8])
def test_operators_on_thin_boxes(cuda_device, N, nel, per):
    wl = _box(nel, N, per)
    wl["S_theta"] = None
    check_nodes(wl, cuda_device)


@pytest.mark.parametrize("shape", sorted(THIN))
def test_restriction_cost_on_thin_boxes(cuda_device, shape):
    """A fine node of a thin box costs at most six times one of a full box (the
    axes' tables are host work by the node of an axis, and the call waits)."""
    import time
    import torch
    from paper_2504_08157_gb300 import xg
    t = {}
    for nel in (THIN[shape], FULL):
        wl = _box(nel)
        with GpuContext(wl) as g, GpuContext(_box(nel, 2)) as c:
            src = torch.from_numpy(wl["q"]).to(cuda_device)
            dst = torch.empty((5, c.np), dtype=torch.float64, device=cuda_device)
            best = float("inf")
            for _ in range(8):
                a = time.perf_counter()
                xg.xg_restrict(g.ctx, c.ctx, src, dst)
                best = min(best, time.perf_counter() - a)
            t[nel] = best / g.np
    assert t[THIN[shape]] <= 6.0 * t[FULL], (t[THIN[shape]] * 1e9, t[FULL] * 1e9)


# (a call's own work, launches and waits, is most of it at 50,000 nodes)
WIDE = {"column": (1, 1, 15600), "pencil": (1, 16000, 4), "sheet": (1, 250, 250)}


@pytest.mark.parametrize("shape", sorted(WIDE))
def test_conservation_sums_cost_on_thin_boxes(cuda_device, shape):
    """A node of a thin box of a million costs at most twice one of a full box."""
    import numpy as np
    t = {}
    for nel in (WIDE[shape], (32, 32, 15)):
        wl = _box(nel)
        with GpuContext(wl) as g:
            t[nel] = _time(lambda: g.xg.xg_diagnostics(g.ctx)) / g.np
            sums = np.array(g.xg.xg_diagnostics(g.ctx))
            m, _, _ = oracle_of(wl)
        M = E.mass(m)
        assert np.all(np.abs(sums - (M * wl["q"]).sum(axis=1)) <= 1e-13 * (M * np.abs(wl["q"])).sum(axis=1))
    assert t[WIDE[shape]] <= 2.0 * t[(32, 32, 15)], t
