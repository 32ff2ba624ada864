"""The workloads whose speed is measured: a user's calls of the solver, from a single small Couette
run to the 2048 x 512 channel, and what each returns in 64 bits.

A case is a dict of plain values.  Every pass hands the library an initial distribution (or fields to
seed it from), takes RK3 steps and reads the result back, all through the public binding.  The
reference part at the end restates the method in plain torch / numpy double precision.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_1708_05944_gb300 import vlb

HH20, HH12, SMALL = "HH(4;8)xH(4;20)", "HH(4;8)xH(4;12)", "HH(3;4)xH(3;4)"


def listed():
    return [
        # the validation run of the paper's first Couette configuration: one small double-precision
        # instance stepped many times, bound by launches and latency
        dict(name="couette_small_fp64", flow="couette", model=SMALL, prec=64, inst=1, cells=32, stretch=0.0,
             steps=12, kn_min=0.1, kn_max=0.1),
        # one ragged single-precision run of the same kind on the scale-up model: a Kn scan's single member
        dict(name="couette_single_fp32", flow="couette", model=HH20, prec=32, inst=1, cells=77, stretch=0.95,
             steps=12, kn_min=0.5, kn_max=0.5),
        # the Couette scale-up: five Knudsen numbers on 1024 cells, tuned, as a production run does
        dict(name="couette_scaleup_fp32", flow="couette", model=HH20, prec=32, inst=5, cells=1024, stretch=0.0,
             steps=12, kn_min=1e-3, kn_max=10.0, tune=True),
        # a ragged batch of 256 instances of 64 .. 1024 cells with a time step each (parameter scan,
        # training data of the warm start)
        dict(name="couette_batch_fp32", flow="couette", model=HH20, prec=32, inst=256, cells=1024, cells_min=64,
             stretch=0.0, steps=3, kn_min=1e-3, kn_max=10.0, tune=True),
        # the double-precision reference solver on the scale-up case
        dict(name="couette_scaleup_fp64", flow="couette", model=HH20, prec=64, inst=5, cells=1024, stretch=0.0,
             steps=3, kn_min=1e-3, kn_max=10.0),
        # seeding from fields, Shakhov collision, fields read back: the warm-started heat-transfer run
        dict(name="couette_shakhov_fp32", flow="couette", model=HH20, prec=32, inst=24, cells=96, cells_min=64,
             stretch=0.0, steps=12, kn_min=0.1, kn_max=10.0, shakhov=True, seeded=True),
        # the conservative f~ formulation on the paper's stretched grid
        dict(name="couette_ftilde_fp32", flow="couette", model=HH20, prec=32, inst=5, cells=1024, stretch=0.95,
             steps=3, kn_min=1e-2, kn_max=10.0, ftilde=True),
        # the ballistic Couette experiment's kind of velocity set (beyond 32 nodes on an axis), few cells
        dict(name="couette_ballistic_fp32", flow="couette", model="HH(4;40)xHH(4;10)", prec=32, inst=1, cells=16,
             stretch=0.95, steps=6, kn_min=1000.0, kn_max=1000.0),
        # the expanding channel at full size: the largest single-GPU configuration
        dict(name="channel_fp32", flow="channel", model=HH12, prec=32, nl=512, nx=2048, steps=1, kn=0.05),
        # the channel's double-precision reference solver
        dict(name="channel_fp64", flow="channel", model=HH12, prec=64, nl=64, nx=256, steps=1, kn=0.05),
        # the Cartesian-split channel the paper compares with
        dict(name="channel_cartesian_fp32", flow="channel", model=HH12, prec=32, nl=256, nx=512, steps=1, kn=0.05,
             cartesian=True),
        # the Poiseuille-limit channel: small velocity set, flow-rate ends, many short steps
        dict(name="channel_flow_small_fp32", flow="channel", model=SMALL, prec=32, nl=16, nx=128, steps=12, kn=0.01,
             q0=0.1),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more workload of the ranges the listed ones stand for."""
    kind = rng.choice(["couette", "couette", "batch", "shakhov", "ftilde", "ballistic", "channel", "channel",
                       "cartesian"])
    prec = rng.choice([32, 32, 32, 64])
    steps = rng.choice([1, 2, 3, 4, 6, 9])
    if kind in ("channel", "cartesian"):
        model = rng.choice([HH12, HH12, SMALL])
        cells = _log(rng, 600, 300_000 if prec == 32 else 30_000)
        nl = max(4, min(512, _log(rng, 8, max(9, cells // 8))))
        c = dict(flow="channel", model=model, prec=prec, nl=nl, nx=4 * max(1, cells // (4 * nl)),
                 steps=min(steps, 3), kn=rng.choice([0.01, 0.05, 0.2, 1.0]))
        if kind == "cartesian":
            c["cartesian"] = True
        elif rng.random() < 0.4:
            c["q0"] = round(rng.uniform(0.02, 0.15), 3)
        return c
    if kind == "ballistic":
        return dict(flow="couette", model="HH(4;%d)xHH(%d;%d)" % (rng.randint(17, 44), 3, rng.randint(4, 10)), prec=prec,
                    inst=rng.choice([1, 2]), cells=rng.randint(8, 48), stretch=rng.choice([0.0, 0.95]), steps=steps,
                    kn_min=10.0, kn_max=1000.0)
    model = rng.choice([HH20, HH20, HH12, SMALL, "HH(3;4)xHH(3;4)", "H(4;6)xHH(3;5)", "HH(2;4)xH(4;8)"])
    total = _log(rng, 40, 60_000 if prec == 32 else 5000)
    inst = _log(rng, 1, max(1, total // 40))
    cells = max(4, total // inst + rng.randint(0, 6))
    if kind in ("shakhov",):
        model = rng.choice([HH20, HH12, SMALL])
    lo, hi = sorted(10.0 ** rng.uniform(-2.5, 1.0) for _ in range(2))
    c = dict(flow="couette", model=model, prec=prec, inst=inst, cells=cells, cells_min=max(4, cells // rng.choice([1, 2, 5])),
             stretch=rng.choice([0.0, 0.0, 0.9, 0.95]), steps=steps, kn_min=lo, kn_max=hi)
    if kind == "shakhov":
        c["shakhov"] = True
        c["seeded"] = rng.random() < 0.5
    elif kind == "ftilde":
        c["ftilde"] = True
    elif kind == "batch":
        c["tune"] = True
    return c


# ------------------------------------------------------------------ the state a user's program holds
def _device():
    return torch.device("cuda")


def _real(case):
    return torch.float64 if case["prec"] == 64 else torch.float32


def _instances(case, seed):
    """Cells, Knudsen number, radii and time step of every instance (the case's own), and its inner
    wall speed (the seed's)."""
    shape, rng = np.random.default_rng([case["inst"], case["cells"]]), np.random.default_rng([seed, 1])
    ax = _axes(case["model"])
    n, p = case["inst"], float(ax[0].p.abs().max())
    kns = np.exp(np.linspace(math.log(case["kn_min"]), math.log(case["kn_max"]), n))
    out = []
    for k in range(n):
        cells = int(shape.integers(case.get("cells_min", case["cells"]), case["cells"] + 1))
        r_out = 2.0 if n <= 8 else float(shape.uniform(1.5, 4.0))
        g = _radial(cells, 1.0, r_out, case["stretch"], 0.5)
        # a quarter of the advection limit, half a relaxation time, and the stability bound of the
        # inertial force (its spectral radius grows with the nodes of both axes)
        rho = float((ax[0].p.abs().max() * ax[1].p.abs().max() * (ax[0].p.abs().max() + ax[1].p.abs().max())))
        dt = min(0.25 * float(g["dr"].min()) / p, 0.3 * 0.6 * float(kns[k]), 0.8 / rho)
        out.append(dict(cells=cells, kn=float(kns[k]), uw=float(rng.uniform(0.01, 0.5)), r_out=r_out, dt=dt))
    return out


def _fields(count, rng, uw):
    """Smooth n, u^0, u^1, T and q^0 across one row of `count` cells: a flow between the walls."""
    s = (torch.arange(count, dtype=torch.float64) + 0.5) / count
    a = torch.tensor(rng.uniform(-1, 1, 5))
    n = 1.0 + 0.05 * a[0] * torch.cos(math.pi * s) + 0.02 * a[1] * torch.sin(3 * s)
    u0 = 0.01 * a[2] * torch.sin(math.pi * s)
    u1 = uw * (1.0 - s) * (1.0 + 0.2 * a[3] * s)
    T = 1.0 + 0.3 * uw * uw * s * (1 - s) + 0.02 * a[4] * torch.sin(2 * s)
    return n, u0, u1, T, 0.01 * torch.sin(math.pi * s) * a[1]


def _rough(shape, seed, amplitude=1e-3):
    """1 + amplitude * U(-1, 1): the noise of a state that has not settled."""
    g = torch.Generator(device=_device())
    g.manual_seed(1000 + seed)
    return 1.0 + amplitude * (2.0 * torch.rand(shape, generator=g, device=_device(), dtype=torch.float32) - 1.0)


def _couette_fields(case, seed):
    rng = np.random.default_rng([seed, 2])
    rows = [_fields(i["cells"], rng, i["uw"]) for i in _instances(case, seed)]
    return [torch.cat([r[k] for r in rows]).to(_device()) for k in range(5)]


def _distribution(case, seed):
    """The initial distribution in the caller's layout and the context's type."""
    ax = _axes(case["model"])
    if case["flow"] == "couette":
        n, u0, u1, T, _ = _couette_fields(case, seed)
    else:
        nl, nx = case["nl"], case["nx"]
        rng = np.random.default_rng([seed, 3])
        a = rng.uniform(-1, 1, 4)
        s = ((torch.arange(nl, dtype=torch.float64, device=_device()) + 0.5) / nl)[None, :]
        x = ((torch.arange(nx, dtype=torch.float64, device=_device()) + 0.5) / nx)[:, None]
        ends = (1.0, 1.0) if "q0" in case else (2.0, 1.0)
        n = (ends[0] + (ends[1] - ends[0]) * x) * (1.0 + 0.02 * a[0] * torch.cos(3 * s + 5 * x))
        u0 = 0.02 * a[1] * torch.sin(math.pi * s) * torch.sin(9 * x)
        u1 = 0.1 * (1.0 + 0.2 * a[2] * torch.cos(4 * x)) * (1.0 - s * s)
        T = 1.0 + 0.02 * a[3] * torch.sin(3 * s) * torch.cos(6 * x)
        n, u0, u1, T = (v.expand(nx, nl).reshape(-1) for v in (n, u0, u1, T))
    out = torch.empty((n.numel(), 2, ax[0].nq, ax[1].nq), dtype=_real(case), device=_device())
    step = max(1, 40_000_000 // (ax[0].nq * ax[1].nq))
    for lo in range(0, n.numel(), step):
        f = _equilibrium(ax, *(v[lo:lo + step] for v in (n, u0, u1, T)))
        out[lo:lo + step] = f * _rough(f.shape, seed * 7919 + lo)
    return out


def _context(case, seed):
    prec = vlb.VLB_FP64 if case["prec"] == 64 else vlb.VLB_FP32_BULK
    if case["flow"] == "channel":
        c = vlb.Channel(case["model"], prec, case["nl"], case["nx"], case["kn"])
        if case.get("cartesian"):
            c.set_formulation(vlb.VLB_CARTESIAN)
        if "q0" in case:
            c.set_flow_rate(case["q0"])
        return c, _channel_dt(case)
    ins = _instances(case, seed)
    c = vlb.Couette(case["model"], prec,
                    [dict(n_cells=i["cells"], r_in=1.0, r_out=i["r_out"], stretch_A=case["stretch"]) for i in ins],
                    [(i["uw"], 1.0) for i in ins], [(0.0, 1.0)] * len(ins), [i["kn"] for i in ins],
                    [vlb.VLB_TAU_AOKI] * len(ins))
    c.set_dt([i["dt"] for i in ins])
    if case.get("ftilde"):
        c.set_formulation(vlb.VLB_FTILDE)
    if case.get("shakhov"):
        c.set_collision(vlb.VLB_SHAKHOV, 2.0 / 3.0)
    if case.get("tune"):
        c.autotune(0.0, reps=5)
    return c, 0.0


def prepare(case, seed):
    ctx, dt = _context(case, seed)
    s = dict(case=case, ctx=ctx, dt=dt, out=torch.empty(ctx.f_shape(), dtype=_real(case), device=_device()))
    if case.get("seeded"):
        s["fields"] = [v.cpu().numpy() for v in _couette_fields(case, seed)]
    else:
        s["f0"] = _distribution(case, seed)
    return s


def run(s):
    """Initial state in, RK3 steps, distribution, wall densities and (seeded runs) fields out.  The
    moments and wall densities of a single-precision run are returned in single precision."""
    case, ctx = s["case"], s["ctx"]
    if "fields" in s:
        ctx.init_from_moments(*s["fields"])
    else:
        ctx.set_f(s["f0"])
    if case["steps"] < 3:
        ctx.step(s["dt"], case["steps"])
    else:
        ctx.step_graph(s["dt"], case["steps"])
    kind = np.float64 if case["prec"] == 64 else np.float32
    out = dict(f=ctx.read_f(s["out"]), nw=ctx.wall_density().astype(kind))
    if "fields" in s:
        n, u0, u1, T, Tab, q = ctx.read_moments(full=True)
        out["moments"] = np.concatenate([np.stack([n, u0, u1, T], 1), Tab, q], 1).astype(kind)
    return out


def work(case):
    """The initial distribution read, the final one written; the arithmetic of every stage."""
    ax = _axes(case["model"])
    v = ax[0].nq * ax[1].nq
    if case["flow"] == "channel":
        cells = case["nl"] * case["nx"]
        contract = 0 if case.get("cartesian") else 2 * (ax[0].nq + ax[1].nq)  # one matrix per axis
        flops = 2 * (2 * 60 + contract // 2 + 30)
    else:
        cells = case["inst"] * (case["cells"] + case.get("cells_min", case["cells"])) // 2
        flops = 2 * (60 + (ax[0].nq + ax[1].nq) + 20)  # half-size blocks of both force matrices
    real = case["prec"] // 8
    given = 5 * 8 * cells if case.get("seeded") else cells * 2 * v * real
    return dict(bytes=float(given + cells * 2 * v * real), flops=float(cells) * v * flops * 3 * case["steps"])


# ------------------------------------------------------------------ the method in 64 bits
class _Axis:
    """Nodes, weights, force matrices and the table of the truncated projection of one axis: the
    half-range rule (positive nodes, then their negatives) or the full-range one, from the
    orthonormal polynomials of exp(-x^2 / 2) / sqrt(2 pi) on the (half) line."""

    def __init__(self, half, N, Q):
        self.half, self.N = half, N
        gx, gw = np.polynomial.legendre.leggauss(48)
        top = 8.0 + 3.0 * math.sqrt(Q)
        edges = np.arange(0.0 if half else -top, top + 1e-9, 0.5)
        x = (edges[:-1, None] + 0.25 * (1.0 + gx[None, :])).ravel().astype(np.longdouble)
        W = np.tile(0.25 * gw, len(edges) - 1) * np.exp(-0.5 * x * x) / np.sqrt(np.longdouble(2.0 * np.pi))
        # Stieltjes: psi_{k+1} b_{k+1} = (x - a_k) psi_k - b_k psi_{k-1}
        psi = [np.ones_like(x) / np.sqrt(W.sum())]
        a, b = [], [np.longdouble(0.0)]
        for k in range(Q):
            a.append((W * x * psi[k] ** 2).sum())
            r = (x - a[k]) * psi[k] - (b[k] * psi[k - 1] if k else 0.0)
            b.append(np.sqrt((W * r * r).sum()))
            psi.append(r / b[-1])

        def values(y, deriv=False):
            v, d = [psi[0][0] * np.ones_like(y)], [np.zeros_like(y)]
            for k in range(Q):
                v.append(((y - a[k]) * v[k] - (b[k] * v[k - 1] if k else 0.0)) / b[k + 1])
                d.append((v[k] + (y - a[k]) * d[k] - (b[k] * d[k - 1] if k else 0.0)) / b[k + 1])
            return (np.array(v), np.array(d)) if deriv else np.array(v)

        J = np.diag(np.array(a, float)) + np.diag(np.array(b[1:Q], float), 1) + np.diag(np.array(b[1:Q], float), -1)
        y = np.linalg.eigvalsh(J).astype(np.longdouble)
        for _ in range(3):
            v, d = values(y, True)
            y = y - v[Q] / d[Q]
        v = values(y)
        w = 1.0 / (v[:Q] ** 2).sum(0)
        # projections of (omega psi_l)' and (p omega psi_l)' on psi_s
        pv, pd = values(x, True)
        pv, pd = pv[:Q], pd[:Q]
        D = (W * pv) @ (pd - x * pv).T
        Dt = (W * pv) @ (pv + x * pd - x * x * pv).T
        if half:
            v0 = values(np.zeros(1, dtype=np.longdouble))[:Q, 0]
            sg = np.repeat([1.0, -1.0], Q)
            vv = np.concatenate([v[:Q], v[:Q]], 1)
            w, p = np.tile(w, 2), np.concatenate([y, -y])
            same = (sg[:, None] == sg[None, :])
            jump = 0.5 / np.sqrt(np.longdouble(2 * np.pi)) * (v0 @ vv)
            K = w[:, None] * (sg[:, None] * same * (vv.T @ D @ vv) + jump[:, None] * sg[None, :] * (v0 @ vv)[None, :])
            Kt = w[:, None] * (same * (vv.T @ Dt @ vv))
        else:
            vv, p = v[:Q], y
            K, Kt = w[:, None] * (vv.T @ D @ vv), w[:, None] * (vv.T @ Dt @ vv)
        # monomial coefficients of psi_l, l <= N, and the table w_k sum_l c_ls psi_l(|p_k|)
        c = np.zeros((N + 1, N + 1), dtype=np.longdouble)
        c[0, 0] = psi[0][0]
        for k in range(N):
            c[k + 1, 1:] += c[k, :-1]
            c[k + 1] -= a[k] * c[k] + (b[k] * c[k - 1] if k else 0.0)
            c[k + 1] /= b[k + 1]
        tab = w[:, None] * (vv[:N + 1].T @ c)
        self.nq = len(p)
        put = lambda z: torch.from_numpy(np.ascontiguousarray(z, dtype=np.float64)).to(_device())
        self.p, self.w, self.K, self.Kt, self.tab = put(p), put(w), put(K), put(Kt), put(tab)

    def project(self, u, T, k=0):
        """Populations (cells, nq) of (p - u)^k times the unit Gaussian of mean u, variance T."""
        N = self.N

        def side(v):  # int_0^inf x^s (x - v)^k N(x; v, T) dx, s = 0 .. N
            M = [0.5 * (1.0 + torch.erf(v / torch.sqrt(2 * T)))]
            M.append(v * M[0] + T * torch.exp(-v * v / (2 * T)) / torch.sqrt(2 * math.pi * T))
            for s in range(2, N + k + 1):
                M.append(v * M[s - 1] + (s - 1) * T * M[s - 2])
            return torch.stack([sum(math.comb(k, i) * (-v) ** (k - i) * M[s + i] for i in range(k + 1))
                                for s in range(N + 1)], 1)

        if self.half:
            q = self.nq // 2
            return torch.cat([side(u) @ self.tab[:q].T, (-1.0) ** k * side(-u) @ self.tab[q:].T], 1)
        central = lambda m: torch.zeros_like(T) if m % 2 else T ** (m // 2) * math.prod(range(m - 1, 0, -2))
        mom = torch.stack([sum(math.comb(s, i) * u ** (s - i) * central(i + k) for i in range(s + 1))
                           for s in range(N + 1)], 1)
        return mom @ self.tab.T


@functools.lru_cache(maxsize=8)
def _axes(model):
    out = []
    for part in model.split("x"):
        kind, rest = part.rstrip(")").split("(")
        N, Q = rest.split(";")
        out.append(_Axis(kind == "HH", int(N), int(Q)))
    return out


def _equilibrium(ax, n, u0, u1, T):
    f = n[:, None, None] * ax[0].project(u0, T)[:, :, None] * ax[1].project(u1, T)[:, None, :]
    return torch.stack([f, T[:, None, None] * f], 1)


def _moments(ax, F):
    """n, u^0, u^1, T of F (cells, 2, nq0, nq1)."""
    p0, p1 = ax[0].p[:, None], ax[1].p[None, :]
    n = F[:, 0].sum((1, 2))
    u0, u1 = (F[:, 0] * p0).sum((1, 2)) / n, (F[:, 0] * p1).sum((1, 2)) / n
    e = ((F[:, 0] * (p0 * p0 + p1 * p1)).sum((1, 2)) + F[:, 1].sum((1, 2))) / n
    return n, u0, u1, (e - u0 * u0 - u1 * u1) / 3.0


def _higher(ax, F, u0, u1):
    x0 = ax[0].p[None, :, None] - u0[:, None, None]
    x1 = ax[1].p[None, None, :] - u1[:, None, None]
    e = 0.5 * (x0 * x0 + x1 * x1) * F[:, 0] + 0.5 * F[:, 1]
    s = lambda v: v.sum((1, 2))
    return s(x0 * x0 * F[:, 0]), s(x0 * x1 * F[:, 0]), s(x1 * x1 * F[:, 0]), s(e * x0), s(e * x1)


def _heat_flux(ax, F, n, u0, u1, T):
    """Grad's heat-flux part for the cell's own q, projected axis by axis."""
    q0, q1 = _higher(ax, F, u0, u1)[3:]
    A = [ax[0].project(u0, T, k)[:, :, None] for k in range(4)]
    B = [ax[1].project(u1, T, k)[:, None, :] for k in range(4)]
    c = lambda v: v[:, None, None]
    t = c(q0) * (A[3] * B[0] + A[1] * B[2]) + c(q1) * (A[2] * B[1] + A[0] * B[3])
    l = c(q0) * A[1] * B[0] + c(q1) * A[0] * B[1]
    iT2 = c(1.0 / (T * T))
    return torch.stack([iT2 * (t / c(5.0 * T) - 0.8 * l), iT2 * (0.2 * t - 0.4 * c(T) * l)], 1)


def _weno(a, b, c, d, e):
    """WENO-5 value right of c, weights delta / sigma^2, vanishing indicators sharing the weight."""
    F1, F2, F3 = a / 3 - 7 * b / 6 + 11 * c / 6, -b / 6 + 5 * c / 6 + d / 3, c / 3 + 5 * d / 6 - e / 6
    s1 = 13 / 12 * (a - 2 * b + c) ** 2 + 0.25 * (a - 4 * b + 3 * c) ** 2
    s2 = 13 / 12 * (b - 2 * c + d) ** 2 + 0.25 * (b - d) ** 2
    s3 = 13 / 12 * (c - 2 * d + e) ** 2 + 0.25 * (3 * c - 4 * d + e) ** 2
    low = torch.minimum(s1, torch.minimum(s2, s3))
    w = []
    for s, delta in ((s1, 0.1), (s2, 0.6), (s3, 0.3)):
        w.append(torch.where(low == 0, (s == 0).to(s.dtype), (low / torch.where(s == 0, torch.ones_like(s), s)) ** 2) * delta)
    return (w[0] * F1 + w[1] * F2 + w[2] * F3) / (w[0] + w[1] + w[2])


def _faces(G, up):
    """Values at the interfaces between cells of G with three ghosts at each end of axis 0; `up`
    says where the velocity is not negative (broadcasts against the result)."""
    n = G.shape[0]
    at = lambda k: G[2 + k:n - 3 + k]
    return torch.where(up, _weno(at(-2), at(-1), at(0), at(1), at(2)), _weno(at(3), at(2), at(1), at(0), at(-1)))


def _radial(n, r_in, r_out, A, delta):
    s, c = np.arange(n + 1), np.arange(n) + 0.5
    if A == 0.0:
        Rf, Rc = r_in + (r_out - r_in) * s / n, r_in + (r_out - r_in) * c / n
        sg, ef, de = Rc.copy(), np.ones(n + 1), (r_out - r_in) / n
    else:
        A0 = max(delta, 1.0 - delta)
        lo, hi = -math.atanh(A * delta / A0), math.atanh(A * (1.0 - delta) / A0)
        de = (hi - lo) / n
        R = lambda eta: r_in + (r_out - r_in) * (delta + A0 / A * np.tanh(eta))
        Rf, Rc = R(lo + s * de), R(lo + c * de)
        Rf[0], Rf[-1] = r_in, r_out
        sg = A0 * (r_out - r_in) * Rc / (A * np.cosh(lo + c * de) ** 2)
        ef = A * np.cosh(lo + s * de) ** 2 / (A0 * (r_out - r_in))
    return dict(Rf=Rf, Rc=Rc, sg=sg, ef=ef, de=de, dr=Rf[1:] - Rf[:-1])


def _couette_rhs(ax, F, g, ins, case, nw):
    p0, p1 = ax[0].p, ax[1].p
    dev = lambda z: torch.from_numpy(z).to(F.device)[:, None, None, None]
    ft = bool(case.get("ftilde"))
    n, u0, u1, T = _moments(ax, F)
    itau = (n / (math.sqrt(math.pi / 8.0) * ins["kn"]))[:, None, None, None]
    target = _equilibrium(ax, n, u0, u1, T)
    if case.get("shakhov"):
        target = target + (1.0 / 3.0) * _heat_flux(ax, F, n, u0, u1, T)
    X = F * dev(g["sg"]) if ft else F
    up = (p0 >= 0)[None, :, None]
    one = torch.ones(1, dtype=torch.float64, device=F.device)
    ends = []
    for k, (E, uw, out) in enumerate(((X[:3], ins["uw"], p0 < 0), (X[-3:].flip(0), 0.0, p0 > 0))):
        out = out[None, :, None]
        g1, g2 = 3 * E[0] - 3 * E[1] + E[2], 6 * E[0] - 8 * E[1] + 3 * E[2]
        flux = (torch.where(out, _weno(E[2], E[1], E[0], g1, g2), 0 * g1)[0] * p0[:, None]).sum()
        wall = _equilibrium(ax, one, 0 * one, uw * one, one)[0]
        nw[k] = -flux / torch.where(out, 0 * wall, wall * p0[:, None])[0].sum()
        inc = nw[k] * wall
        ends.append([torch.where(out, x, inc) for x in (g1, g2, g2)])
    G = torch.cat([torch.stack(ends[0][::-1]), X, torch.stack(ends[1])])
    V = _faces(G, up)
    if ft:
        ef = dev(g["ef"])
        adv = p0[:, None] * (ef[1:] * V[1:] - ef[:-1] * V[:-1]) / (g["de"] * dev(g["sg"]))
        R = dev(g["Rc"])
    else:
        Rf = dev(g["Rf"])
        adv = p0[:, None] * (Rf[1:] * V[1:] - Rf[:-1] * V[:-1]) / (0.5 * (Rf[1:] ** 2 - Rf[:-1] ** 2))
        R = 0.5 * (Rf[1:] + Rf[:-1])
    force = (p1 ** 2 * torch.matmul(ax[0].K, F) - p0[:, None] * torch.matmul(F, ax[1].Kt.T)) / R
    return -adv - force - (F - target) * itau


def _phi(x):
    return 0.5 * (math.tanh(2.0) - np.tanh(2.0 - 0.3 * x)), 0.15 / np.cosh(2.0 - 0.3 * x) ** 2


def _channel_grid(case):
    nl, nx, A = case["nl"], case["nx"], 0.95
    top = math.atanh(A)
    lf, lc = np.tanh(np.arange(nl + 1) / nl * top) / A, np.tanh((np.arange(nl) + 0.5) / nl * top) / A
    lf[-1] = 1.0
    xf, xc = -10.0 + 50.0 * np.arange(nx + 1) / nx, -10.0 + 50.0 * (np.arange(nx) + 0.5) / nx
    chi = (1.0 + math.tanh(2.0) / 2.0) * xf + 100.0 / 60.0 * np.log(np.cosh(2.0 - 0.3 * xf) / math.cosh(2.0))
    return dict(lf=lf, lc=lc, xf=xf, xc=xc, dl=lf[1:] - lf[:-1], dchi=chi[1:] - chi[:-1])


def _channel_dt(case):
    g, ax = _channel_grid(case), _axes(case["model"])
    p = max(float(a.p.abs().max()) for a in ax)
    return min(0.2 * min(g["dl"].min(), g["dchi"].min()) / p, 0.1 * case["kn"], 2e-3)


def _channel_rhs(ax, F, case, g, nw):
    """F: (nx, nl, 2, nq0, nq1), the caller's order."""
    nx, nl = case["nx"], case["nl"]
    p0, p1 = ax[0].p, ax[1].p
    P0, P1 = p0[:, None], p1[None, :]
    clb = bool(case.get("cartesian"))
    dev = lambda z: torch.from_numpy(np.ascontiguousarray(z)).to(F.device)
    b4 = lambda z: z[..., None, None, None]
    one = torch.ones(1, dtype=torch.float64, device=F.device)
    L = torch.empty_like(F)
    lf, lc = g["lf"], g["lc"]
    ph, dp = _phi(g["xc"])
    phf, dpf = _phi(g["xf"])
    a = np.sqrt(1.0 + lf[None, :] ** 2 * dp[:, None] ** 2) / (1.0 + ph[:, None])
    root = np.sqrt(1.0 + lc[None, :] ** 2 * dpf[:, None] ** 2)
    b = (1.0 + phf)[:, None] / root
    c = lc[None, :] * dpf[:, None] * (1.0 + phf)[:, None] / root
    glxl = (b[1:] - b[:-1]) / g["dchi"][:, None]
    glxx = -(a[:, 1:] - a[:, :-1]) / g["dl"][None, :] + (c[1:] - c[:-1]) / g["dchi"][:, None]
    wall = _equilibrium(ax, one, 0 * one, 0 * one, one)[0]
    mirror = torch.arange(ax[0].nq, device=F.device).roll(ax[0].nq // 2)
    ends_u = []
    # columns: moments, collision, force, lambda advection
    for lo in range(0, nx, max(1, 60_000_000 // (nl * 2 * ax[0].nq * ax[1].nq))):
        hi = min(nx, lo + max(1, 60_000_000 // (nl * 2 * ax[0].nq * ax[1].nq)))
        X = F[lo:hi]
        flat = X.reshape(-1, *X.shape[2:])
        n, u0, u1, T = _moments(ax, flat)
        R = -(flat - _equilibrium(ax, n, u0, u1, T)) * b4(n * T / case["kn"])
        if not clb:
            gx, gl = (b4(dev(z[lo:hi]).reshape(-1)) for z in (glxx, glxl))
            R += gx * (P1 ** 2 * torch.matmul(ax[0].K, flat) - P0 * torch.matmul(flat, ax[1].Kt.T))
            R -= gl * (P0 ** 2 * torch.matmul(flat, ax[1].K.T) - P1 * torch.matmul(ax[0].Kt, flat))
        ends_u.append(u1.reshape(hi - lo, nl)[[0, -1]])
        Y = X.transpose(0, 1)
        af = dev(a[lo:hi].T.copy())
        if clb:
            ia = dev(1.0 / (1.0 + ph[lo:hi]))
            V = b4(ia[None, :] * torch.ones(nl + 1, 1, device=F.device, dtype=F.dtype)) * (
                P0 - b4(dev(lf)[:, None] * dev(dp[lo:hi])[None, :]) * P1)
        else:
            V = b4(af) * P0 + 0 * P1
        out = V[nl] > 0
        E = Y[-3:].flip(0)
        g1, g2 = 3 * E[0] - 3 * E[1] + E[2], 6 * E[0] - 8 * E[1] + 3 * E[2]
        flux = (torch.where(out, _weno(E[2], E[1], E[0], g1, g2) * V[nl], 0 * g1))[:, 0].sum((1, 2))
        den = torch.where(out, 0 * wall, wall * V[nl])[:, 0].sum((1, 2))
        nw[lo:hi] = -flux / den
        inc = b4(nw[lo:hi]) * wall
        top = [torch.where(out, x, inc) for x in (g1, g2, g2)]
        G = torch.cat([Y[:3].flip(0)[:, :, :, mirror], Y, torch.stack(top)])
        fl = V * _faces(G, V >= 0)
        R = R.reshape(X.shape) - ((fl[1:] - fl[:-1]) / b4(dev(g["dl"])[:, None])).transpose(0, 1)
        L[lo:hi] = R
    u_in, u_out = ends_u[0][0], ends_u[-1][1]
    # rows: xi advection
    step = max(1, 30_000_000 // (nx * 2 * ax[0].nq * ax[1].nq))
    for lo in range(0, nl, step):
        hi = min(nl, lo + step)
        X = F[:, lo:hi]
        if clb:
            V = b4(dev(1.0 + phf)[:, None]) * P1 + 0 * P0
            V = V.expand(nx + 1, hi - lo, 1, ax[0].nq, ax[1].nq)
        else:
            V = b4(dev(b[:, lo:hi])) * P1 - b4(dev(c[:, lo:hi])) * P0
        T0 = torch.ones(hi - lo, dtype=torch.float64, device=F.device)
        side = []
        for k, (ur, nres, adj, Ve, into) in enumerate(((u_in, 2.0, X[0], V[0], V[0] > 0), (u_out, 1.0, X[-1], V[-1], V[-1] < 0))):
            if "q0" in case:
                pe = _phi(g["xf"][0 if k == 0 else -1])[0]
                Q = dev(1.5 * case["q0"] * (1.0 - lc[lo:hi] ** 2) / (1.0 + pe))
                f1 = _equilibrium(ax, T0, 0 * T0, Q, T0)
                leaving = torch.where(into, 0 * adj, Ve * adj)[:, 0].sum((1, 2))
                entering = torch.where(into, Ve * f1, 0 * f1)[:, 0].sum((1, 2))
                f = b4(((1.0 + pe) * Q - leaving) / entering) * f1
            else:
                f = nres * _equilibrium(ax, T0, 0 * T0, ur[lo:hi], T0)
            side.append(torch.where(into, f, adj))
        G = torch.cat([side[0][None].expand(3, *side[0].shape), X, side[1][None].expand(3, *side[1].shape)])
        fl = V * _faces(G, V >= 0)
        L[:, lo:hi] -= (fl[1:] - fl[:-1]) / b4(dev(g["dchi"])[:, None])
    return L


def _rk3(F, dt, steps, rhs):
    for _ in range(steps):
        F1 = F + dt * rhs(F)
        F2 = 0.75 * F + 0.25 * F1 + 0.25 * dt * rhs(F1)
        F = F / 3.0 + 2.0 / 3.0 * F2 + 2.0 / 3.0 * dt * rhs(F2)
    return F


def exact(case, seed):
    ax = _axes(case["model"])
    if case["flow"] == "channel":
        shape = (case["nx"], case["nl"], 2, ax[0].nq, ax[1].nq)
        F = _distribution(case, seed).double().reshape(shape)
        nw = torch.zeros(case["nx"], dtype=torch.float64, device=_device())
        g = _channel_grid(case)
        F = _rk3(F, _channel_dt(case), case["steps"], lambda X: _channel_rhs(ax, X, case, g, nw))
        return dict(f=F.reshape(-1, *shape[2:]), nw=nw.cpu().numpy())
    ins = _instances(case, seed)
    if case.get("seeded"):
        n, u0, u1, T, q = _couette_fields(case, seed)
        F = _equilibrium(ax, n, u0, u1, T)
        A = [ax[0].project(u0, T, k)[:, :, None] for k in range(4)]
        B = [ax[1].project(u1, T, k)[:, None, :] for k in range(4)]
        c = lambda v: v[:, None, None]
        t3, t1 = A[3] * B[0] + A[1] * B[2], A[1] * B[0]
        F = F + c(q / T ** 2)[:, None] * torch.stack([t3 / c(5 * T) - 0.8 * t1, 0.2 * t3 - 0.4 * c(T) * t1], 1)
    else:
        F = _distribution(case, seed).double()
    nw = torch.zeros(len(ins), 2, dtype=torch.float64, device=_device())
    out, at = torch.empty_like(F), 0
    for k, i in enumerate(ins):
        g = _radial(i["cells"], 1.0, i["r_out"], case["stretch"], 0.5)
        sl = slice(at, at + i["cells"])
        out[sl] = _rk3(F[sl], i["dt"], case["steps"], lambda X: _couette_rhs(ax, X, g, i, case, nw[k]))
        at += i["cells"]
    res = dict(f=out, nw=nw.cpu().numpy())
    if case.get("seeded"):
        n, u0, u1, T = _moments(ax, out)
        res["moments"] = torch.stack([n, u0, u1, T, *_higher(ax, out, u0, u1)], 1).cpu().numpy()
    return res
