"""GPU checks of what the fixed-point contractions (xg_fixed.cuh) owe to each
node, whatever the rest of its tile, its line or the other direction holds: a
constant has no derivative at all, and an error is one of the values in the
node's own element segments."""

import numpy as np
import pytest

from inputs import workloads as W
from oracle import euler as E, lgl

from helpers import GpuContext, oracle_of

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


# A node's error is compared with sum_d R_d max |F_d|, over the directions, with
# R_d the largest row sum of the line's matrix and the maximum over the node's
# own segments.  A flux carries up to eight FP64 roundings of 2^-53 (1/rho,
# u, theta, the pressure, their products), a row, the sums over the directions,
# the level's coefficients and the result up to eight more; the fixed-point rows
# 2^-58 of the same.
TOL = 16 * 2.0 ** -53


class Lines:
    """Assembled 1-D operators of a box in extended precision.  Along the
    direction ``uniform`` the box's fields do not vary, and nothing is allowed
    for it."""

    def __init__(self, wl, uniform=None):
        self.wl, self.N, self.uniform = wl, wl["N"], uniform
        self.n = [wl["N"] * e + (0 if p else 1) for e, p in zip(wl["nel"], wl["periodic"])]
        x = lgl.lgl_points_extended(self.N)
        self.D, self.w = lgl.derivative_matrix(x), lgl.lgl_weights(self.N, x)
        self.h = [(np.longdouble(b) - a) / e for a, b, e in zip(wl["lo"], wl["hi"], wl["nel"])]

    def field(self, a):
        return np.asarray(a, dtype=np.longdouble).reshape(self.n[::-1])

    def level(self, a):
        return np.asarray(a, dtype=np.longdouble)[:, None, None]

    def rows(self, M, f, d):
        """(sum of the node's rows of M along d, R max |f| over its segments)."""
        if d == self.uniform:
            return np.zeros_like(f), np.zeros_like(f)
        f = np.moveaxis(f, 2 - d, -1)
        N, nel, per = self.N, self.wl["nel"][d], self.wl["periodic"][d]
        out, top = np.zeros_like(f), np.zeros_like(f)
        R = np.abs(M).sum(axis=1).max()
        for s in range(nel):
            k = (s * N + np.arange(N + 1)) % f.shape[-1]
            seg = f[..., k]
            r = (seg[..., None, :] * M).sum(axis=-1)
            if not per and s == 0:
                r[..., 0] *= 2
            if not per and s == nel - 1:
                r[..., N] *= 2
            for a in range(N + 1):   # a periodic line of one segment meets itself
                out[..., k[a]] += r[..., a]
                top[..., k[a]] = np.maximum(top[..., k[a]], R * np.abs(seg).max(axis=-1))
        return np.moveaxis(out, -1, 2 - d), np.moveaxis(top, -1, 2 - d)

    def derivative(self, f, d):
        M = -(2 / self.h[d]) * self.D
        M[[0, -1]] /= 2
        return self.rows(M, f, d)

    def laplacian(self, f, nu):
        out, top = 0, 0
        for d in range(3):
            K = (self.w[:, None, None] * self.D[:, :, None] * self.D[:, None, :]).sum(axis=0)
            wa = self.w.copy()
            wa[[0, -1]] *= 2
            o, t = self.rows(-nu[d] * (2 / self.h[d]) ** 2 * K / wa[:, None], f, d)
            out, top = out + o, top + t
        return out, top

    def walls(self, L):
        for d in range(3):
            if not self.wl["periodic"][d]:
                np.moveaxis(L[1 + d], 2 - d, 0)[[0, -1]] = 0
        return L

    def rhs(self, q, phys):
        q = [self.field(v) for v in q]
        r0, T0 = self.level(self.wl["rho0"]), self.level(self.wl["Theta0"])
        F = E.fluxes(r0 + 0 * q[0], T0 + 0 * q[0], q, phys)
        L, top = [0] * 5, [0] * 5
        for v in range(5):
            for d in range(3):
                o, t = self.derivative(F[v][d], d)
                L[v], top[v] = L[v] + o, top[v] + t
        g, f = np.longdouble(phys.g), np.longdouble(phys.f)
        for v, a in ((1, f * q[2]), (2, -f * q[1]), (3, -g * q[0])):
            L[v], top[v] = L[v] + a, top[v] + np.abs(a)
        return self.walls(L), top

    def linear(self, v, phys):
        v = [self.field(a) for a in v]
        r0, T0 = self.level(self.wl["rho0"]), self.level(self.wl["Theta0"])
        th0, p = T0 / r0, phys.gamma * E.pressure(T0, phys) / T0 * v[4]
        div = [self.derivative(v[1 + d], d) for d in range(3)]
        A = (div[0][0] + div[1][0], div[0][1] + div[1][1])
        grad = [self.derivative(p, d) for d in range(3)]
        tz = self.derivative(th0 * v[3], 2)
        gr = np.longdouble(phys.g) * v[0]
        L = [A[0] + div[2][0], grad[0][0], grad[1][0], grad[2][0] - gr, th0 * A[0] + tz[0]]
        top = [A[1] + div[2][1], grad[0][1], grad[1][1], grad[2][1] + np.abs(gr), th0 * A[1] + tz[1]]
        return self.walls(L), top


def _beyond(got, ref, top):
    """The largest error in units of a node's allowance."""
    got = np.asarray(got, dtype=np.longdouble).reshape(ref.shape)
    return float((np.abs(got - ref) / (TOL * top + np.longdouble(1e-300))).max())


def _check(wl, device, uniform=None):
    """Tendency, linear operator and hyper-diffusion of wl's state, node by
    node; the mixed form's rho' and Theta' too."""
    import torch
    ref, (_, phys, _) = Lines(wl, uniform), oracle_of(wl)
    L, top = ref.rhs(wl["q"], phys)
    worst = {}
    for prec, vs in ((0, range(5)), (2, (0, 4))):
        with GpuContext(wl, precision=prec) as g:
            got = g.rhs()
        for v in vs:
            worst["rhs", prec, v] = _beyond(got[v], L[v], top[v])
    with GpuContext(wl) as g:
        t = torch.from_numpy(wl["q"]).to(device)
        out = torch.empty_like(t)
        g.xg.xg_linear_operator(g.ctx, t, out)
        got = out.cpu().numpy()
        L, top = ref.linear(wl["q"], phys)
        for v in range(5):
            worst["linear", v] = _beyond(got[v], L[v], top[v])
        g.xg.xg_set_dynamics(g.ctx, (1e-4, 1e-4, 1e-4), 0.5, 0.0, 0.0)
        g.xg.xg_dynamics_tendency(g.ctx, out)
        got = out.cpu().numpy()
    nu = [np.sqrt(np.longdouble(1e-4)) * (h / wl["N"]) ** 2 / np.sqrt(np.longdouble(0.5)) for h in ref.h]
    for v in range(5):
        first, t1 = ref.laplacian(ref.field(wl["q"][v]), nu)
        second, t2 = ref.laplacian(first, nu)
        worst["hyper", v] = _beyond(got[v], -second, t2 + ref.laplacian(t1, nu)[1])   # and the first pass's error
    assert max(worst.values()) <= 1.0, {k: w for k, w in worst.items() if w > 1.0}


@pytest.mark.parametrize("fall", [0, 1])
@pytest.mark.parametrize("per", [(False, True, False), (True, False, True)])
@pytest.mark.parametrize("N", [1, 3, 4, 5, 8])
def test_quiet_nodes_keep_their_digits(cuda_device, N, per, fall):
    """A state that falls by 2^-60 along x or y (2^-4 to 2^-15 an element), so
    that every tile holds loud and quiet nodes."""
    nel = {1: (40, 34, 2), 3: (11, 12, 2), 4: (9, 10, 2), 5: (7, 7, 2), 8: (4, 5, 1)}[N]
    wl = W.box(nel, N, (0.0, 0.0, 0.0), (1000.0 * nel[0], 800.0 * nel[1], 500.0 * nel[2]), per, f=1.0e-4, seed=23)
    wl["S_theta"] = None
    n = [N * e + (0 if p else 1) for e, p in zip(nel, per)]
    s = np.exp2(-60.0 * np.linspace(0.0, 1.0, n[fall]))
    k = np.arange(wl["q"].shape[1])
    wl["q"] = wl["q"] * s[k % n[0] if fall == 0 else k // n[0] % n[1]]
    _check(wl, cuda_device)


@pytest.mark.parametrize("uniform", [True, False])
@pytest.mark.parametrize("narrow,ratio", [(0, 1e3), (1, 1e3), (0, 1e5), (1, 1e5), (2, 1e5)])
@pytest.mark.parametrize("N", [2, 4, 5, 7])
def test_spacings_of_different_size(cuda_device, N, narrow, ratio, uniform):
    """One direction's spacing 1e3 and 1e5 times smaller than the others': the
    wide directions' derivatives keep FP64's precision, which shows where the
    state does not vary along the narrow one."""
    nel, h = (4, 3, 2), [2000.0, 2000.0, 2000.0]
    h[narrow] /= ratio
    per = (True, True, False)
    wl = W.box(nel, N, (0.0, 0.0, 0.0), tuple(n * d for n, d in zip(nel, h)), per, f=1.0e-4, seed=19)
    wl["S_theta"] = None
    if uniform:
        if narrow == 2:
            pytest.skip("the reference state varies along z")
        n = [N * e + (0 if p else 1) for e, p in zip(nel, per)]
        q = wl["q"].reshape([5] + n[::-1])
        wl["q"] = np.ascontiguousarray(np.broadcast_to(q.take([1], axis=3 - narrow), q.shape)).reshape(5, -1)
    _check(wl, cuda_device, narrow if uniform else None)


@pytest.mark.parametrize("off", [(0,), (1,), (2,), (0, 1), (1, 2), (0, 2)])
@pytest.mark.parametrize("N,nel", [(4, (9, 9, 2)), (5, (7, 6, 2)), (4, (1, 6, 5)), (1, (33, 32, 2))])
def test_diffusion_off_in_some_directions(cuda_device, N, nel, off):
    """A direction without diffusion takes nothing from the others' rows, weak
    diffusion's included (its matrix is small against one)."""
    import torch
    wl = W.box(nel, N, (0.0, 0.0, 0.0), (9.0e4 * nel[0], 8.0e4 * nel[1], 7.0e3 * nel[2]), (True, False, False), seed=43)
    c = [0.0 if d in off else 1e-18 for d in range(3)]     # the axes are in the order of their spacing
    ref = Lines(wl)
    with GpuContext(wl) as g:
        g.xg.xg_set_dynamics(g.ctx, tuple(c), 0.5, 0.0, 0.0)
        out = torch.empty((5, g.np), dtype=torch.float64, device=cuda_device)
        g.xg.xg_dynamics_tendency(g.ctx, out)
        got = out.cpu().numpy()
    nu = [np.sqrt(np.longdouble(a)) * (h / N) ** 2 / np.sqrt(np.longdouble(0.5)) for a, h in zip(c, ref.h)]
    for v in range(5):
        first, t1 = ref.laplacian(ref.field(wl["q"][v]), nu)
        second, t2 = ref.laplacian(first, nu)
        assert _beyond(got[v], -second, t2 + ref.laplacian(t1, nu)[1]) <= 1.0
