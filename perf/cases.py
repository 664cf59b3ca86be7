"""What is measured when this framework is timed: the calls its users make,
over the sizes they make them at.

Every case goes through the public entry points of
``paper_2504_08157_gb300.xg``.  Sizes come from the named workloads of
``inputs.workloads`` (the rising bubble, the cyclone box, the paper's timing
grid, the batch of limited-area boxes, the learned closure's box) and the
ragged boxes of the parity tests; the inputs are sampled here, on the GPU,
with the recipes of ``inputs.atmosphere`` and a seeded smooth perturbation.

``exact`` evaluates the same quantities in FP64 with plain torch operations
(element gather, derivative matrix, weighted assembly), sharing nothing with
the library.
"""

import math

import numpy as np
import torch

from paper_2504_08157_gb300 import xg

G, R_D, CP, CV, P_A = 9.81, 287.0, 1004.5, 717.5, 1.0e5
GAMMA = CP / CV
PRECISION = {"fp64": xg.XG_FP64, "df64": xg.XG_DF64, "fp32": xg.XG_FP32}
DEV = "cuda"
BATCH_BOX = (512.0e3, 512.0e3, 20.0e3)


# ------------------------------------------------------------------ the cases

def listed():
    return [
        # a forecast of the 10 km rising-bubble box: the smallest mesh in use,
        # ten steps between outputs
        dict(name="bubble_steps", kind="steps", box="bubble", precision="df64", order=4, nx=8, ny=8, nz=8,
             steps=10),
        # one tendency of an odd box of high order with walls in x and z: a
        # user's own time integrator, or a parity check, around xg_rhs
        dict(name="ragged_rhs", kind="rhs", box="ragged", precision="fp64", order=7, nx=11, ny=6, nz=5,
             per_x=False, per_y=True),
        # the cyclone box at full size in the FP64-accurate mixed precision
        dict(name="cyclone_df64", kind="steps", box="cyclone", precision="df64", order=4, nx=128, ny=128, nz=16,
             steps=1),
        # the same in the FP32 precision form
        dict(name="cyclone_fp32", kind="steps", box="cyclone", precision="fp32", order=4, nx=128, ny=128, nz=16,
             steps=2),
        # native FP64 explicit steps with the paper's hyper-diffusion and sponge
        dict(name="dynamics_fp64", kind="dynamics", box="cyclone", order=4, nx=64, ny=64, nz=16, steps=1),
        # the paper's own timing run: its Table 1 grid, integrator and step
        dict(name="paper_imex", kind="imex", box="paper", order=5, nx=80, ny=80, nz=24),
        # 96 uneven limited-area boxes advanced together
        dict(name="ensemble_batch", kind="batch", count=96, steps=4),
        # a coarse run with the learned closure in every stage
        dict(name="closure_step", kind="closure", box="closure", order=4, nx=64, ny=64, nz=16, steps=1),
        # one Adam update of the closure's training (closure.train's minibatch)
        dict(name="closure_train", kind="train", samples=4096),
        # one snapshot of the closure's training data: the restricted state's
        # features, and the two tendencies that its target is the difference of
        dict(name="closure_data", kind="data", order=4, nx=64, ny=64, nz=16),
        # the intensity diagnostics written with every output of the cyclone box
        dict(name="cyclone_monitor", kind="monitor", box="cyclone", precision="df64", order=4, nx=128, ny=128,
             nz=16, strips=50),
        # independent states streamed from and to host memory
        dict(name="stream_df64", kind="stream", box="cyclone", precision="df64", order=4, nx=32, ny=32, nz=16,
             count=6, steps=1),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _mesh(rng, most_nodes, order, nz_range):
    """Element counts with about most_nodes^u nodes, uneven in x and y."""
    nz = rng.randint(*nz_range)
    n = math.exp(rng.uniform(math.log(2000.0), math.log(most_nodes)))
    side = max(1.0, math.sqrt(n / (order ** 3 * nz)))
    skew = math.exp(rng.uniform(-0.5, 0.5))
    nx, ny = max(1, int(side * skew)), max(1, int(side / skew))
    return dict(order=order, nx=nx, ny=ny, nz=nz)


def draw(rng):
    kind = rng.choice(["steps", "steps", "steps", "rhs", "rhs", "dynamics", "imex", "batch", "closure", "train",
                       "data", "monitor", "stream"])
    if kind == "steps":
        return dict(kind=kind, box=rng.choice(["bubble", "cyclone", "cyclone"]),
                    precision=rng.choice(["fp64", "df64", "fp32"]), steps=rng.randint(1, 4),
                    **_mesh(rng, 4.0e6, rng.randint(3, 6), (3, 24)))
    if kind == "rhs":
        return dict(kind=kind, box="ragged", precision=rng.choice(["fp64", "df64", "fp32"]),
                    per_x=rng.random() < 0.5, per_y=rng.random() < 0.5,
                    **_mesh(rng, 4.0e6, rng.randint(1, 8), (1, 12)))
    if kind == "dynamics":
        return dict(kind=kind, box="cyclone", steps=rng.randint(1, 2),
                    **_mesh(rng, 2.0e6, rng.randint(3, 6), (3, 24)))
    if kind == "imex":
        return dict(kind=kind, box="paper", **_mesh(rng, 2.0e6, rng.randint(3, 6), (4, 24)))
    if kind == "batch":
        return dict(kind=kind, count=_log(rng, 4, 96), steps=rng.randint(1, 4))
    if kind == "closure":
        return dict(kind=kind, box="closure", steps=rng.randint(1, 2),
                    **_mesh(rng, 2.0e6, rng.randint(3, 5), (4, 16)))
    if kind == "train":
        return dict(kind=kind, samples=_log(rng, 300, 200000))
    if kind == "data":
        return dict(kind=kind, **_mesh(rng, 1.0e6, rng.randint(3, 5), (4, 16)))
    if kind == "monitor":
        return dict(kind=kind, box="cyclone", precision=rng.choice(["fp64", "df64", "fp32"]),
                    strips=rng.choice([20, 50, 100]), **_mesh(rng, 4.0e6, 4, (8, 24)))
    return dict(kind=kind, box="cyclone", precision=rng.choice(["fp64", "df64"]), count=rng.randint(2, 6),
                steps=rng.randint(1, 2), **_mesh(rng, 1.0e6, 4, (4, 16)))


# ------------------------------------------------------------------ meshes and fields

def _lgl(N):
    """LGL points, weights and derivative matrix of order N (FP64)."""
    P = np.polynomial.legendre
    c = np.zeros(N + 1)
    c[N] = 1.0
    x = np.array([-1.0, 1.0]) if N == 1 else np.concatenate(([-1.0], np.sort(np.real(P.legroots(P.legder(c)))), [1.0]))
    for _ in range(3):   # polish the interior roots of P_N'
        d1, d2 = P.legval(x, P.legder(c)), P.legval(x, P.legder(c, 2))
        x[1:-1] -= d1[1:-1] / d2[1:-1]
    pn = P.legval(x, c)
    w = 2.0 / (N * (N + 1) * pn ** 2)
    D = np.zeros((N + 1, N + 1))
    for i in range(N + 1):
        for j in range(N + 1):
            if i != j:
                D[i, j] = pn[i] / (pn[j] * (x[i] - x[j]))
    D[0, 0], D[N, N] = -N * (N + 1) / 4.0, N * (N + 1) / 4.0
    return x, w, D


def _box(case):
    """Geometry and physics of a case's box: nel, N, lo, hi, periodic, f, dt
    (the explicit step of the named workload, at its vertical spacing)."""
    N, nel = case["order"], (case["nx"], case["ny"], case["nz"])
    box = case.get("box", "closure")
    if box in ("bubble", "closure"):
        lo, hi, per, f = (0.0, 0.0, 0.0), (10.0e3,) * 3, (False, False, False), 0.0
    elif box == "cyclone":   # the cyclone box's element size
        hx, hy = 8.0e3 * nel[0], 8.0e3 * nel[1]
        lo, hi, per, f = (-hx / 2, -hy / 2, 0.0), (hx / 2, hy / 2, 20.0e3), (True, True, False), 5.0e-5
    elif box == "paper":     # the paper's grid: 10 km elements
        hx, hy = 1.0e4 * nel[0], 1.0e4 * nel[1]
        lo, hi, per, f = (-hx / 2, -hy / 2, 0.0), (hx / 2, hy / 2, 20.0e3), (True, True, False), 5.0e-5
    else:                    # ragged: 1 km elements
        lo, hi = (0.0, 0.0, 0.0), tuple(1.0e3 * n for n in nel)
        per, f = (bool(case["per_x"]), bool(case["per_y"]), False), 1.0e-4
    x, _, _ = _lgl(N)
    dmin = min((hi[d] - lo[d]) / nel[d] * (x[1] - x[0]) / 2.0 for d in range(3))
    return dict(nel=nel, N=N, lo=lo, hi=hi, per=per, f=f, dt=0.1 * dmin / 216.0, box=box)


def _axes(b):
    out = []
    x, _, _ = _lgl(b["N"])
    for d in range(3):
        n = b["N"] * b["nel"][d] + (0 if b["per"][d] else 1)
        g = np.arange(n)
        e = np.minimum(g // b["N"], b["nel"][d] - 1)
        a = g - b["N"] * e
        h = (b["hi"][d] - b["lo"][d]) / b["nel"][d]
        out.append(b["lo"][d] + (e + (x[a] + 1.0) / 2.0) * h)
    return out


def _sounding(z, box):
    if box in ("bubble", "closure"):       # isentropic
        th = np.full_like(z, 300.0)
        pi0 = 1.0 - G * z / (CP * 300.0)
    else:                                  # constant Brunt-Vaisala frequency 0.01 1/s
        s = 1.0e-4 / G
        th = 300.0 * np.exp(s * z)
        pi0 = 1.0 + G * G / (CP * 300.0 * 1.0e-4) * (np.exp(-s * z) - 1.0)
    rho0 = P_A * pi0 ** (CP / R_D) / (R_D * pi0 * th)
    return rho0, rho0 * th


def _t(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to(DEV)


def _fields(b, seed, vmax=15.0, rmax=50.0e3):
    """(q [5, Np], rho0, Theta0, S [Np]) on the GPU: the box's vortex (and in
    the 10 km boxes its warm bubble), a seeded smooth perturbation of every
    variable as a run develops within minutes, and the heating."""
    rng = np.random.RandomState(seed % (2 ** 31))
    ax = _axes(b)
    X, Y, Z = (_t(a) for a in ax)
    nz, ny, nx = Z.numel(), Y.numel(), X.numel()
    rho0, Th0 = _sounding(ax[2] - b["lo"][2], b["box"])
    r0, t0 = _t(rho0), _t(Th0)
    q = torch.zeros((5, nz, ny, nx), dtype=torch.float64, device=DEV)
    L = [b["hi"][d] - b["lo"][d] for d in range(3)]
    s = [(a - b["lo"][d]) / L[d] for d, a in enumerate((X, Y, Z))]
    for v, amp in enumerate((2e-3, 1.0, 1.0, 0.5, 0.3)):
        for _ in range(3):
            k, ph = rng.randint(1, 4, 3), 2.0 * math.pi * rng.rand(3)
            a = amp * (0.5 + rng.rand()) / 3.0
            m = [torch.sin(2.0 * math.pi * int(k[d]) * s[d] + float(ph[d])) for d in range(3)]
            if 1 <= v <= 3 and not b["per"][v - 1]:
                m[v - 1] = m[v - 1] * torch.sin(math.pi * s[v - 1])
            q[v] += (a * m[2])[:, None, None] * (m[1][:, None] * m[0][None, :])[None]
    small = b["box"] != "cyclone" and b["box"] != "paper" and b["box"] != "batch"
    c = [(b["lo"][d] + b["hi"][d]) / 2.0 + L[d] * 0.05 * (rng.rand() - 0.5) for d in range(2)]
    rm, D1, D2 = (0.15 * min(L[:2]), 4.0e3, 0.35 * min(L[:2])) if small else \
        (min(rmax, 0.1 * min(L[:2])), 5823.0, min(200.0e3, 0.25 * min(L[:2])))
    vm = (5.0 if small else vmax) * (0.8 + 0.4 * rng.rand())
    dx, dy = X[None, :] - c[0], Y[:, None] - c[1]
    r = torch.sqrt(dx * dx + dy * dy).clamp_min(1e-30)
    ut = torch.where(r <= rm, vm * r / rm, vm * torch.sqrt(rm / r)) * torch.exp(-(r / D2) ** 6) / r
    hz = r0 * torch.exp(-((Z - b["lo"][2]) / D1) ** 2 / 2.0)
    edge = [torch.ones_like(X), torch.ones_like(Y)]
    for d in range(2):
        if not b["per"][d]:
            edge[d] = torch.sin(math.pi * s[d])
    env = edge[1][:, None] * edge[0][None, :]
    q[1] -= hz[:, None, None] * (ut * dy * env)[None]
    q[2] += hz[:, None, None] * (ut * dx * env)[None]
    if b["box"] in ("bubble", "closure"):   # +1..3 K cosine bubble, Exner pressure unperturbed
        dth, rad, zc = 1.0 + 2.0 * rng.rand(), 1.5e3 + 1.0e3 * rng.rand(), 2.0e3 + 1.0e3 * rng.rand()
        rr = torch.sqrt(dx[None] ** 2 + dy[None] ** 2 + (Z[:, None, None] - zc) ** 2)
        thp = torch.where(rr <= rad, 0.5 * dth * (1.0 + torch.cos(math.pi * rr / rad)), torch.zeros_like(rr))
        q[0] += (r0[:, None, None] * 300.0) / (300.0 + thp) - r0[:, None, None]
    for d in range(3):                      # no flux through the walls
        if not b["per"][d]:
            w = q[1 + d].transpose(0, 2 - d)
            w[0] = 0.0
            w[-1] = 0.0
    ring, width = (0.2 * min(L[:2]), 0.05 * min(L[:2])) if small else (0.8 * rm, 1.0e4)
    S = 10.0 * torch.exp(-((r - ring) / width) ** 2)
    if not small:
        for _ in range(16):
            rc, phi, amp = 2.0e4 + 1.0e5 * rng.rand(), 2.0 * math.pi * rng.rand(), 5.0 + 15.0 * rng.rand()
            S = S + amp * torch.exp(-((dx - rc * math.cos(phi)) ** 2 + (dy - rc * math.sin(phi)) ** 2) / 2.5e7)
    zz = Z - b["lo"][2]
    S = torch.where(zz <= 15.0e3, torch.sin(math.pi * zz.clamp(0.0, 15.0e3) / 15.0e3),
                    torch.zeros_like(zz))[:, None, None] * S[None] / 3600.0
    return q.reshape(5, -1).contiguous(), r0, t0, S.reshape(-1).contiguous()


class _Handle:
    """A context or batch that goes with the state that holds it."""

    def __init__(self, h, free=xg.xg_destroy):
        self.h, self._free = h, free

    def __del__(self):
        if self.h:
            self._free(self.h)
            self.h = None


def _desc(b, precision):
    return xg.mesh_desc(b["nel"], b["N"], b["lo"], b["hi"], b["per"], f=b["f"], g=G, R=R_D, cp=CP, cv=CV, p_a=P_A,
                        precision=PRECISION[precision])


def _context(b, precision, fields, forced=True):
    q, r0, t0, S = fields
    c = _Handle(xg.xg_mesh_create(_desc(b, precision)))
    xg.xg_set_state(c.h, q, r0, t0)
    if forced:
        xg.xg_set_forcing(c.h, S)
    return c


def _batch_boxes(count):
    """Seeded limited-area boxes of the batched form: 4..24 elements
    horizontally, 4..12 vertically, orders 3..6.  The sizes do not depend on
    the case's seed (a program's ensemble keeps its meshes)."""
    rng = np.random.RandomState(4096)
    out = []
    for i in range(count):
        nel = (rng.randint(4, 25), rng.randint(4, 25), rng.randint(4, 13))
        N = int(rng.randint(3, 7))
        b = dict(nel=tuple(int(n) for n in nel), N=N, lo=(-BATCH_BOX[0] / 2, -BATCH_BOX[1] / 2, 0.0),
                 hi=(BATCH_BOX[0] / 2, BATCH_BOX[1] / 2, BATCH_BOX[2]), per=(True, True, False), f=5.0e-5,
                 box="batch")
        x, _, _ = _lgl(N)
        b["dt"] = 0.1 * BATCH_BOX[2] / b["nel"][2] * (x[1] - x[0]) / 2.0 / 216.0
        b["vmax"], b["rmax"] = 10.0 + 20.0 * rng.rand(), 30.0e3 + 50.0e3 * rng.rand()
        out.append(b)
    return out


def _network(seed):
    """A trained-looking network: parameters, then the input mean and scale
    and the output scale that training derives from its samples."""
    g = torch.Generator(device="cpu").manual_seed(seed % (2 ** 31))
    p = []
    for fin, fout in ((21, 64), (64, 64), (64, 5)):
        p.append((2.0 * torch.rand(fin * fout, generator=g) - 1.0) / math.sqrt(fin))
        p.append(0.1 * (2.0 * torch.rand(fout, generator=g) - 1.0))
    return torch.cat(p).to(torch.float32).to(DEV)


def _feature_scales():
    """Typical size of the 21 features (the state, its gradients, the heating)
    and of the five targets in the closure's box."""
    s = np.array([2e-3, 1.0, 1.0, 0.5, 0.3])
    scale = np.concatenate([s, np.repeat(s, 3) * 1e-3, [1e-3]])
    return scale, s * 1e-5


# ------------------------------------------------------------------ prepare and run

def prepare(case, seed):
    kind = case["kind"]
    st = dict(case=case)
    if kind == "batch":
        boxes = _batch_boxes(case["count"])
        st["dt"] = np.array([b["dt"] for b in boxes])
        st["batch"] = _Handle(xg.xg_batch_create([_desc(b, "fp32") for b in boxes]), xg.xg_batch_destroy)
        st["inst"], st["q"] = [], []
        n = 0
        for i, b in enumerate(boxes):
            q, r0, t0, S = _fields(b, seed + 7919 * i, b["vmax"], b["rmax"])
            h = xg.xg_batch_instance(st["batch"].h, i)
            xg.xg_set_state(h, q, r0, t0)
            xg.xg_set_forcing(h, S)
            st["inst"].append(h)
            st["q"].append(q)
            n += q.numel()
        flat = torch.empty(n, dtype=torch.float64, device=DEV)
        st["flat"], st["out"], o = flat, [], 0
        for q in st["q"]:
            st["out"].append(flat[o:o + q.numel()].view_as(q))
            o += q.numel()
        return st
    if kind == "train":
        n = case["samples"]
        g = torch.Generator(device=DEV).manual_seed(seed % (2 ** 31))
        scale, out = _feature_scales()
        mix = torch.randn(5, 21, generator=g, device=DEV) / 5.0
        Z = torch.randn(21, n, generator=g, device=DEV)
        st["X"] = (Z * _t(scale.astype(np.float32))[:, None]).contiguous()
        noise = torch.randn(5, n, generator=g, device=DEV)
        st["T"] = ((mix @ torch.tanh(Z) + 0.5 * noise) * _t(out.astype(np.float32))[:, None]).contiguous()
        st["mean"] = torch.zeros(21, device=DEV)
        st["scale"], st["oscale"] = _t((1.0 / scale).astype(np.float32)), _t(out.astype(np.float32))
        # Adam in mid-training: moments of the size of the gradients
        p = _network(seed)
        st["p0"], st["m0"] = p, 1e-3 * torch.randn(p.numel(), generator=g, device=DEV)
        st["v0"] = 1e-6 * (0.5 + torch.rand(p.numel(), generator=g, device=DEV))
        st["p"], st["m"], st["v"], st["g"] = (torch.empty_like(p) for _ in range(4))
        return st
    b = st["b"] = _box(case)
    if kind == "data":
        fine = dict(b, nel=tuple(2 * n for n in b["nel"]))
        f = _fields(fine, seed)
        st["fine"] = _context(fine, "fp32", f)
        rho0, Th0 = _sounding(_axes(b)[2] - b["lo"][2], b["box"])
        c = st["coarse"] = _Handle(xg.xg_mesh_create(_desc(b, "fp32")))
        npc = xg.xg_mesh_np(c.h)
        st["qc"], st["rcf"], st["rc"] = (torch.zeros((5, npc), dtype=torch.float64, device=DEV) for _ in range(3))
        xg.xg_set_state(c.h, st["qc"], _t(rho0), _t(Th0))
        st["qf"], st["rf"] = f[0], torch.empty_like(f[0])
        st["X"] = torch.empty((21, npc), dtype=torch.float32, device=DEV)
        return st
    f = _fields(b, seed)
    precision = {"dynamics": "fp64", "imex": "fp64", "closure": "fp32"}.get(kind) or case["precision"]
    c = st["ctx"] = _context(b, precision, f)
    st["q"], st["precision"] = f[0], precision
    if kind in ("dynamics", "imex"):
        xg.xg_set_dynamics(c.h, (1e-4, 1e-4, 1e-4), 0.5, 4000.0, 0.05)
    if kind == "closure":
        scale, out = _feature_scales()
        xg.xg_closure_set(c.h, _network(seed), torch.zeros(21, device=DEV), _t((1.0 / scale).astype(np.float32)),
                          _t(out.astype(np.float32)))
    if kind == "stream":
        n = case["count"]
        pin = dict(dtype=torch.float64, pin_memory=True)
        st["in"], st["out"] = [], [torch.empty(f[0].shape, **pin) for _ in range(n)]
        for k in range(n):
            h = torch.empty(f[0].shape, **pin)
            h.copy_(f[0] * (1.0 - 0.05 * k))
            st["in"].append(h)
        del st["q"]
        return st
    st["out"] = torch.empty_like(f[0])
    return st


def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "batch":
        for h, q in zip(st["inst"], st["q"]):
            xg.xg_set_state(h, q)
        xg.xg_batch_step(st["batch"].h, st["dt"], case["steps"])
        for h, o in zip(st["inst"], st["out"]):
            xg.xg_get_state(h, o)
        return st["flat"].to(torch.float32)
    if kind == "train":
        st["p"].copy_(st["p0"])
        st["m"].copy_(st["m0"])
        st["v"].copy_(st["v0"])
        loss = xg.xg_mlp_loss_grad(st["p"], st["X"], st["T"], st["mean"], st["scale"], st["oscale"], st["g"])
        xg.xg_mlp_adam(st["p"], st["m"], st["v"], st["g"], 100, lr=2e-3)
        return dict(loss=torch.tensor(loss, dtype=torch.float32), grad=st["g"], params=st["p"], m=st["m"], v=st["v"])
    if kind == "data":
        fine, coarse = st["fine"].h, st["coarse"].h
        xg.xg_restrict(fine, coarse, st["qf"], st["qc"])
        xg.xg_set_state(coarse, st["qc"])
        xg.xg_features(coarse, st["X"])
        xg.xg_rhs(fine, st["rf"])
        xg.xg_restrict(fine, coarse, st["rf"], st["rcf"])
        xg.xg_rhs(coarse, st["rc"])
        return dict(X=st["X"], fine=st["rcf"].to(torch.float32), coarse=st["rc"].to(torch.float32))
    c = st["ctx"].h
    if kind == "stream":
        xg.xg_step_stream(c, st["in"], st["out"], st["b"]["dt"], case["steps"])
        return list(st["out"])
    if kind == "monitor":
        sums = xg.xg_diagnostics(c)
        u, cent, means = xg.xg_ri_velocity(c, case["strips"])
        return dict(sums=np.array(sums), u_ri=np.array([u]), centroid=cent, means=means)
    xg.xg_set_state(c, st["q"])
    if kind == "rhs":
        xg.xg_rhs(c, st["out"])
    else:
        if kind == "imex":
            xg.xg_step_imex(c, 0.5, 1)
        else:
            xg.xg_step(c, st["b"]["dt"], case["steps"])
        xg.xg_get_state(c, st["out"])
    return st["out"].to(torch.float32) if st["precision"] == "fp32" else st["out"]


# ------------------------------------------------------------------ work

def _np(b):
    return math.prod(b["N"] * b["nel"][d] + (0 if b["per"][d] else 1) for d in range(3))


def work(case):
    """Compulsory bytes and operations of one pass.  A stage reads the state
    (and the heating, and q^n in stages 2-3) and writes the new one: 88, 128
    and 128 bytes a node in 8-byte values; the copies into and out of the
    context read and write 40 bytes a node each (FP32 contexts convert, and
    the output is narrowed)."""
    kind = case["kind"]
    if kind == "train":
        n, p = case["samples"], xg.XG_CLOSURE_PARAMS
        return dict(bytes=4 * (26 * n + 8 * p), flops=6.0 * p * n)
    if kind == "batch":
        boxes = _batch_boxes(case["count"])
        return dict(bytes=sum(_np(b) * (172 * case["steps"] + 180) for b in boxes),
                    flops=sum(_np(b) * 3 * (150 + 40 * b["N"]) * case["steps"] for b in boxes))
    b = _box(case)
    n, N = _np(b), b["N"]
    flops = n * (150 + 40 * N)           # one tendency: pointwise work and three contractions of five variables
    if kind == "data":
        nf = _np(dict(b, nel=tuple(2 * k for k in b["nel"])))
        return dict(bytes=nf * (40 + 24 + 40) + n * (40 + 84 + 24 + 40 + 40 + 40),
                    flops=flops * 9 + 2 * 5 * nf * 2 * (N + 1))
    if kind == "monitor":
        width = 4 if case["precision"] == "fp32" else 8
        return dict(bytes=n * 5 * width, flops=n * 40)
    value = 4 if {"closure": "fp32"}.get(kind, case.get("precision")) == "fp32" else 8
    copies = 180 if value == 4 else 160
    if kind == "rhs":
        return dict(bytes=n * (80 + (60 + 44 if value == 4 else 88)), flops=flops)
    if kind == "stream":
        return dict(bytes=case["count"] * n * (80 + 43 * value * case["steps"]),
                    flops=case["count"] * case["steps"] * 3 * flops)
    if kind == "imex":   # three tendencies with hyper-diffusion, and two solves of about ten operator products
        return dict(bytes=n * (160 + 3 * 168 + 2 * 10 * 80), flops=3 * flops + n * 20 * (14 * N + 100))
    extra_b, extra_f = (0, 0)
    if kind == "dynamics":
        extra_f = 3 * n * 2 * 5 * 3 * 2 * (N + 1)
    if kind == "closure":
        extra_f = 3 * n * (2 * xg.XG_CLOSURE_PARAMS + 15 * 2 * (N + 1))
    return dict(bytes=n * (copies + 43 * value * case["steps"] + extra_b),
                flops=case["steps"] * (3 * flops + extra_f))


# ------------------------------------------------------------------ 64-bit values

class _Exact:
    """The assembled operators of a box in FP64: every line of nodes is
    gathered into element segments, multiplied by the 1-D matrix, weighted and
    summed at shared nodes."""

    def __init__(self, b, r0, t0, S):
        self.b, self.S = b, S
        self.n = [b["N"] * b["nel"][d] + (0 if b["per"][d] else 1) for d in range(3)]
        x, w, D = _lgl(b["N"])
        self.h = [(b["hi"][d] - b["lo"][d]) / b["nel"][d] for d in range(3)]
        self.w, self.D = _t(w), _t(D)
        self.K = self.D.T @ (self.w[:, None] * self.D)
        self.idx, self.W = [], []
        for d in range(3):
            i = (torch.arange(b["nel"][d], device=DEV)[:, None] * b["N"]
                 + torch.arange(b["N"] + 1, device=DEV)[None, :]) % self.n[d]
            self.idx.append(i.reshape(-1))
            self.W.append(torch.zeros(self.n[d], dtype=torch.float64, device=DEV).index_add_(
                0, i.reshape(-1), self.w.repeat(b["nel"][d])))
        self.r0, self.t0 = r0[:, None, None], t0[:, None, None]
        self.p0 = P_A * (R_D * self.t0 / P_A) ** GAMMA

    def line(self, f, d, M):
        """Assembled (weighted) 1-D operator: sum_e (M f_e) / W along d."""
        dim = f.dim() - 1 - d
        e = f.index_select(dim, self.idx[d]).movedim(dim, -1)
        e = (e.reshape(e.shape[:-1] + (-1, self.b["N"] + 1)) @ M.T).flatten(-2).movedim(-1, dim)
        out = torch.zeros_like(f).index_add_(dim, self.idx[d], e)
        return out / self.W[d].reshape([-1] + [1] * d)

    def dx(self, f, d):
        return (2.0 / self.h[d]) * self.line(f, d, self.w[:, None] * self.D)

    def walls(self, L):
        for d in range(3):
            if not self.b["per"][d]:
                w = L[1 + d].transpose(0, 2 - d)
                w[0] = 0.0
                w[-1] = 0.0
        return L

    def view(self, q):
        return q.view(-1, self.n[2], self.n[1], self.n[0])

    def rhs(self, q, extra=None):
        q = self.view(q)
        rho, th = self.r0 + q[0], self.t0 + q[4]
        pp = self.p0 * torch.expm1(GAMMA * torch.log1p(q[4] / self.t0))
        L = torch.zeros_like(q)
        for d in range(3):
            u = q[1 + d] / rho
            F = torch.stack([q[1 + d], q[1] * u, q[2] * u, q[3] * u, th * u])
            F[1 + d] += pp
            L -= self.dx(F, d)
            del F
        L[1] += self.b["f"] * q[2]
        L[2] -= self.b["f"] * q[1]
        L[3] -= G * q[0]
        if self.S is not None:
            L[4] += rho * self.S.view_as(rho)
        if extra is not None:
            L += self.view(extra(q))
        return self.walls(L).reshape(5, -1)

    def step(self, q, dt, extra=None):
        q1 = q + dt * self.rhs(q, extra)
        q2 = 0.75 * q + 0.25 * (q1 + dt * self.rhs(q1, extra))
        return q / 3.0 + (2.0 / 3.0) * (q2 + dt * self.rhs(q2, extra))

    def dynamics(self, q):
        """Hyper-diffusion (c = 1e-4, 0.5 s) and the 4 km sponge of 0.05 1/s."""
        q = self.view(q)
        lap = lambda f: sum(-(math.sqrt(1e-4) * (self.h[d] / self.b["N"]) ** 2 / math.sqrt(0.5))  # noqa: E731
                            * (2.0 / self.h[d]) ** 2 * self.line(f, d, self.K) for d in range(3))
        E = torch.stack([-lap(lap(q[v])) for v in range(5)])
        z = _t(_axes(self.b)[2])
        a = ((z - (self.b["hi"][2] - 4000.0)) / 4000.0).clamp(0.0, 1.0)
        E[3] -= (0.05 * torch.sin(0.5 * math.pi * a) ** 2)[:, None, None] * q[3]
        return E

    def linear(self, v):
        v = self.view(v)
        c = GAMMA * self.p0 / self.t0
        th0 = self.t0 / self.r0
        L = torch.zeros_like(v)
        dxu, dyv = -self.dx(v[1], 0), -self.dx(v[2], 1)
        L[0] = dxu + dyv - self.dx(v[3], 2)
        L[1], L[2] = -c * self.dx(v[4], 0), -c * self.dx(v[4], 1)
        L[3] = -self.dx(c * v[4], 2) - G * v[0]
        L[4] = th0 * (dxu + dyv) - self.dx(th0 * v[3], 2)
        return self.walls(L).reshape(5, -1)

    def solve(self, h, rhs, x):
        """(I - h L) x = rhs by GMRES to 1e-13, variables scaled to unit size."""
        sc = rhs.square().mean(dim=1, keepdim=True).sqrt().clamp_min(1e-300)
        A = lambda v: v - h * self.linear(v * sc) / sc  # noqa: E731
        bs, x = rhs / sc, x / sc
        bn = float(bs.norm())
        for _ in range(4):
            r = bs - A(x)
            beta = float(r.norm())
            if beta <= 1e-13 * bn:
                break
            V, H = [r / beta], np.zeros((41, 40))
            for j in range(40):
                w = A(V[j])
                for _ in range(2):
                    for i, v in enumerate(V):
                        a = float(torch.dot(v.view(-1), w.view(-1)))
                        H[i, j] += a
                        w = w - a * v
                H[j + 1, j] = float(w.norm())
                V.append(w / H[j + 1, j])
                e = np.zeros(j + 2)
                e[0] = beta
                y, _, _, _ = np.linalg.lstsq(H[:j + 2, :j + 1], e, rcond=None)
                if np.linalg.norm(H[:j + 2, :j + 1] @ y - e) <= 1e-14 * bn:
                    break
            for i, a in enumerate(y):
                x = x + float(a) * V[i]
            del V
        return x * sc

    def imex(self, q, dt):
        """ARK2 of Giraldo, Kelly & Constantinescu (2013): one step."""
        g, dl = 1.0 - 1.0 / math.sqrt(2.0), 1.0 / (2.0 * math.sqrt(2.0))
        al = (3.0 + 2.0 * math.sqrt(2.0)) / 6.0
        ae, ai, bw = ((), (2 * g,), (1 - al, al)), ((), (g,), (dl, dl)), (dl, dl, g)
        S, Lq, x = [self.rhs(q, self.dynamics)], [self.linear(q)], q
        for i in (1, 2):
            r = q + dt * sum(ae[i][j] * (S[j] - Lq[j]) + ai[i][j] * Lq[j] for j in range(i))
            x = self.solve(dt * g, r, x)
            S.append(self.rhs(x, self.dynamics))
            Lq.append(self.linear(x))
        return q + dt * sum(bw[j] * S[j] for j in range(3))

    def features(self, q):
        q = self.view(q)
        rows = [q[v] for v in range(5)] + [self.dx(q[v], d) for v in range(5) for d in range(3)]
        rows.append(self.S.view_as(q[0]) if self.S is not None else torch.zeros_like(q[0]))
        return torch.stack([r.reshape(-1) for r in rows])


def _mlp(p, Z):
    """The network of normalised, clamped inputs Z [21, n] in FP64."""
    o = 0
    for i, (fin, fout) in enumerate(((21, 64), (64, 64), (64, 5))):
        W, o = p[o:o + fin * fout].view(fout, fin), o + fin * fout
        Z, o = W @ Z + p[o:o + fout, None], o + fout
        if i < 2:
            Z = Z * torch.sigmoid(Z)
    return Z


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        return None          # 96 boxes one after the other take too long
    with torch.no_grad():
        if kind == "train":
            st = prepare(case, seed)
            f64 = lambda k: st[k].double()  # noqa: E731
            Z = ((f64("X") - f64("mean")[:, None]) * f64("scale")[:, None]).clamp(-8.0, 8.0)
            T = f64("T") / f64("oscale")[:, None]
            p = f64("p0").requires_grad_(True)
            with torch.enable_grad():
                loss = (_mlp(p, Z) - T).square().mean()
                g, = torch.autograd.grad(loss, p)
            m, v = 0.9 * f64("m0") + 0.1 * g, 0.999 * f64("v0") + 0.001 * g * g
            new = f64("p0") - 2e-3 * (m / (1.0 - 0.9 ** 100)) / ((v / (1.0 - 0.999 ** 100)).sqrt() + 1e-8)
            return dict(loss=loss.detach(), grad=g, params=new, m=m, v=v)
        b = _box(case)
        if kind == "data":
            fine = dict(b, nel=tuple(2 * n for n in b["nel"]))
            qf, r0, t0, S = _fields(fine, seed)
            ef = _Exact(fine, r0, t0, S)
            rho0, Th0 = _sounding(_axes(b)[2] - b["lo"][2], b["box"])
            ec = _Exact(b, _t(rho0), _t(Th0), None)

            def restrict(f):
                f = ef.view(f)
                for d in range(3):
                    dim = 3 - d
                    f = (f.movedim(dim, -1) @ _restriction(fine, b, d).T).movedim(-1, dim)
                return f.reshape(f.shape[0], -1).contiguous()

            qc = restrict(qf)
            return dict(X=ec.features(qc), fine=restrict(ef.rhs(qf)), coarse=ec.rhs(qc))
        q, r0, t0, S = _fields(b, seed)
        e = _Exact(b, r0, t0, S)
        if kind == "rhs":
            return e.rhs(q)
        if kind == "monitor":
            return _monitor(e, b, q, r0, case["strips"])
        if kind == "stream":
            out = []
            for k in range(case["count"]):
                x = q * (1.0 - 0.05 * k)
                for _ in range(case["steps"]):
                    x = e.step(x, b["dt"])
                out.append(x)
            return out
        if kind == "imex":
            return e.imex(q, 0.5)
        extra = None
        if kind == "dynamics":
            extra = e.dynamics
        if kind == "closure":
            scale, osc = _feature_scales()
            p, sc = _network(seed).double(), _t(1.0 / scale)[:, None]
            extra = lambda x: _mlp(p, (e.features(x) * sc).clamp(-8.0, 8.0)) * _t(osc)[:, None]  # noqa: E731
        for _ in range(case["steps"]):
            q = e.step(q, b["dt"], extra)
        return q


def _restriction(fine, coarse, d):
    """Dense 1-D matrix of the fine elements' interpolants at the coarse nodes."""
    x, _, _ = _lgl(fine["N"])
    xc, _, _ = _lgl(coarse["N"])
    nf = fine["N"] * fine["nel"][d] + (0 if fine["per"][d] else 1)
    nc = coarse["N"] * coarse["nel"][d] + (0 if coarse["per"][d] else 1)
    M = np.zeros((nc, nf))
    for g in range(nc):
        e = min(g // coarse["N"], coarse["nel"][d] - 1)
        s = (e + (xc[g - coarse["N"] * e] + 1.0) / 2.0) / coarse["nel"][d] * fine["nel"][d]
        k = max(0, min(int(math.floor(s)), fine["nel"][d] - 1))
        t = 2.0 * (s - k) - 1.0
        for a in range(fine["N"] + 1):
            M[g, (fine["N"] * k + a) % nf] += math.prod((t - x[j]) / (x[a] - x[j]) for j in range(fine["N"] + 1)
                                                        if j != a)
    return _t(M)


def _monitor(e, b, q, r0, strips):
    q = e.view(q)
    J = math.prod(h / 2.0 for h in e.h)
    M = J * e.W[2][:, None, None] * e.W[1][None, :, None] * e.W[0][None, None, :]
    sums = torch.stack([(M * q[v]).sum() for v in range(5)])
    X, Y, _ = (_t(a) for a in _axes(b))
    rho = r0[:, None, None] + q[0]
    u, v, w = q[1] / rho, q[2] / rho, q[3] / rho
    sp = torch.sqrt(u * u + v * v + w * w)
    tot = sp.sum(dim=(1, 2))
    cent = torch.stack([(sp * X[None, None, :]).sum(dim=(1, 2)) / tot, (sp * Y[None, :, None]).sum(dim=(1, 2)) / tot],
                       dim=1)
    R = 0.5 * min(b["hi"][d] - b["lo"][d] for d in range(2))
    dx = X[None, None, :] - cent[:, 0, None, None]
    dy = Y[None, :, None] - cent[:, 1, None, None]
    r = torch.sqrt(dx * dx + dy * dy)
    ut = (u * (-dy) + v * dx).abs() / r.clamp_min(1e-300)
    k = torch.floor(r / (R / strips)).clamp_max(strips).long()
    k = k + (strips + 1) * torch.arange(k.shape[0], device=DEV)[:, None, None]
    n = (strips + 1) * q.shape[1]
    cnt = torch.bincount(k.reshape(-1), minlength=n).view(-1, strips + 1)[:, :strips]
    s = torch.bincount(k.reshape(-1), weights=ut.reshape(-1), minlength=n).view(-1, strips + 1)[:, :strips]
    means = torch.where(cnt > 0, s / cnt.clamp_min(1), torch.zeros_like(s))
    return dict(sums=sums, u_ri=means.max().reshape(1), centroid=cent, means=means)
