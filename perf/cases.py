"""Performance cases of the CMCG Helmholtz solver: one pass each through its public entry points.

A case is a dict of plain values; ``listed`` gives the fixed ones, ``draw`` more of the same
ranges, ``prepare`` the solver handle and the device inputs a user's program holds before the
call, ``run`` the call, ``work`` the bytes and operations one pass cannot do without, and
``exact`` the same result in plain torch, 64-bit.

The problems are those of the repository's workloads: a 2D Gaussian source in a homogeneous
medium, the uneven 2D batch's smooth random media, a square sound-soft obstacle, scattering of a
plane wave off a sound-soft sphere in 3D, and the 3D layered medium (4th order).  Everything is
generated on the GPU from the seed.  Fields handed to a period are superpositions of plane waves
at the problem's wavenumber, which is what CG directions and mismatches look like.
"""
from __future__ import annotations

import math

import torch

from paper_1903_12522_gb300 import cmcg

DEV = "cuda"
F64 = torch.float64
PREC = {"fp64": cmcg.FP64, "fp32": cmcg.FP32}


def listed():
    return [
        # the smallest call: one forced period on the 2D Gaussian workload's grid; launches and
        # latency are everything (a user stepping a small 2D problem, or a served 2D request)
        dict(name="wave2d_small_f32", op="wave", medium="gauss", prec="fp32", order=2, nx=128, ny=128, nz=0),
        # backward period in the default precision on a ragged 2D grid with a sound-soft obstacle
        # (the gradient evaluations of the obstacle studies)
        dict(name="adjoint2d_ragged_f64", op="adjoint", medium="square", prec="fp64", order=2, nx=436, ny=301, nz=0),
        # the largest member of the uneven 2D batch: heterogeneous medium, 1025^2 nodes
        dict(name="wave2d_large_f32", op="wave", medium="random", prec="fp32", order=2, nx=1024, ny=1024, nz=0),
        # the flagship: one forced period of the 257^3 sphere-scattering workload in FP32
        dict(name="wave3d_f32", op="wave", medium="sphere", prec="fp32", order=2, nx=256, ny=256, nz=256),
        # backward period on a ragged mid-size 3D box, odd sizes in every axis
        dict(name="adjoint3d_ragged_f32", op="adjoint", medium="sphere", prec="fp32", order=2, nx=149, ny=96, nz=122),
        # one forced period in the default precision on a 3D grid larger than the L2 cache
        # (outer gradients, FP64 reference solves)
        dict(name="wave3d_f64", op="wave", medium="sphere", prec="fp64", order=2, nx=192, ny=192, nz=192),
        # 4th-order stencil on the layered medium with interior point sources
        dict(name="wave3d_order4_f32", op="wave", medium="layered", prec="fp32", order=4, nx=256, ny=256, nz=256),
        # the exact Riesz map (FP64 multigrid PCG), once per CG iteration of a default solve
        dict(name="riesz3d", op="riesz", medium="sphere", prec="fp64", order=2, nx=128, ny=128, nz=128),
        # first-order (staggered) formulation: one forced period
        dict(name="fo_wave3d_f32", op="fo_wave", medium="sphere", prec="fp32", order=2, nx=128, ny=128, nz=128),
        # a whole solve with default options (FP64, exact Riesz map), within an iteration budget
        dict(name="solve2d_f64", op="solve", medium="gauss", prec="fp64", order=2, nx=128, ny=128, nz=0, iters=8),
        # a whole solve as production runs it in 3D: FP32 periods, one V-cycle per iteration as
        # Riesz map, run-up, kappa held in L2; an iteration budget bounds the pass
        dict(name="solve3d_f32_vcycle", op="solve", medium="sphere", prec="fp32", order=2, nx=96, ny=96, nz=96,
             iters=8, vcycle=True, runup=2),
        # six uneven 2D requests through the multi-solve engine
        dict(name="engine2d_f32", op="engine", medium="random", prec="fp32", order=2, nx=384, ny=384, nz=0, iters=5,
             slots=6),
    ]


def _size(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["wave", "adjoint", "wave", "adjoint", "riesz", "fo_wave", "fo_adjoint", "solve", "engine"])
    dim = rng.choice([2, 3])
    prec = rng.choice(["fp32", "fp64"])
    order = 2
    if op in ("wave", "adjoint"):
        order = rng.choice([2, 2, 4])
        if dim == 2:
            n = [_size(rng, 64, 1024) for _ in range(2)]
        else:
            n = [_size(rng, 32, 256 if prec == "fp32" else 176) for _ in range(3)]
    elif op == "riesz":
        prec = "fp64"
        n = [_size(rng, 64, 768) for _ in range(2)] if dim == 2 else [_size(rng, 32, 144) for _ in range(3)]
    elif op in ("fo_wave", "fo_adjoint"):
        n = [_size(rng, 64, 768) for _ in range(2)] if dim == 2 else [_size(rng, 32, 144 if prec == "fp32" else 96)
                                                                    for _ in range(3)]
    elif op == "solve":
        n = [_size(rng, 64, 320) for _ in range(2)] if dim == 2 else [_size(rng, 32, 104) for _ in range(3)]
    else:
        dim, prec = 2, "fp32"
        m = _size(rng, 96, 512)
        n = [m, m]
    if order == 4:
        medium = "random" if dim == 2 else "layered"  # the 4th-order stencil takes no Dirichlet nodes
    elif dim == 2:
        medium = rng.choice(["gauss", "random", "square"])
    else:
        medium = rng.choice(["sphere", "sphere", "layered"])
    if op == "engine":
        medium = "random"
    case = dict(op=op, medium=medium, prec=prec, order=order, nx=n[0], ny=n[1], nz=n[2] if dim == 3 else 0)
    if op == "solve":
        case["iters"] = rng.randint(4, 10)
        if prec == "fp32":
            case["vcycle"] = True
            case["runup"] = rng.randint(0, 3)
    if op == "engine":
        case["iters"] = rng.randint(3, 6)
        case["slots"] = rng.randint(2, 6)
    return case


# ---- the problem of a case -------------------------------------------------------------------
def _coords(n, h):
    d = len(n)
    return [(torch.arange(n[a] + 1, device=DEV, dtype=F64) * h).reshape([-1 if b == d - 1 - a else 1 for b in range(d)])
            for a in range(d)]


class _Problem:
    """Medium, frequency, mask, sources and initial data of one case, made from the seed."""

    def __init__(self, case, seed, salt=0):
        gen = torch.Generator()
        gen.manual_seed(1000003 * (int(seed) + 1) + salt)

        def uni(lo, hi, k=1):
            return (lo + (hi - lo) * torch.rand(k, generator=gen, dtype=F64)).tolist()

        n = [case["nx"], case["ny"]] + ([case["nz"]] if case["nz"] else [])
        self.n, self.d = tuple(n), len(n)
        self.h = h = 1.0 / max(n)
        self.ext = [m * h for m in n]
        self.shape = tuple(m + 1 for m in reversed(n))
        self.order, self.medium = case["order"], case["medium"]
        xs = _coords(n, h)
        one = torch.ones(self.shape, device=DEV, dtype=F64)
        self.faces = (cmcg.BC_ABC,) * 4 + ((cmcg.BC_ABC,) * 2 if self.d == 3 else (cmcg.BC_NEUMANN,) * 2)
        self.mask = self.f = self.g = None
        centre = [e * u for e, u in zip(self.ext, uni(0.35, 0.65, self.d))]
        r2 = sum((x - c0) ** 2 for x, c0 in zip(xs, centre))
        if self.medium == "gauss":  # homogeneous, 16 points per wavelength, dt = h/2
            self.c, ppw, c_min, self.dt = one, 16.0, 1.0, 0.5 * h
            self.f = torch.exp(-r2 / (2 * 0.05 ** 2))
        elif self.medium == "square":  # plane wave on a sound-soft square, dt = 0.4 h
            self.c, ppw, c_min, self.dt = one, 12.8, 1.0, 0.4 * h
            inside = one > 0
            for x, c0, e in zip(xs, centre, self.ext):
                inside = inside & (torch.abs(x - c0) <= 0.15 * e)
            self.mask = inside.to(torch.uint8)
        elif self.medium == "random":  # smooth medium in [1, 2], one source
            f = sum(torch.sin(sum(2 * math.pi * k * x for k, x in zip(uni(-4, 4, self.d), xs)) + uni(0, 6.28)[0])
                    for _ in range(6)) * one
            self.c = 1.0 + (f - f.min()) / (f.max() - f.min())
            ppw, c_min = 8.0 + 12.0 * ((sum(n) * 7919) % 1000) / 1000.0, 1.0
            self.dt = 0.9 * h / (math.sqrt(self.d) * 2.0)
            if self.order == 4:
                self.dt *= math.sqrt(0.75)
            self.f = torch.exp(-r2 / (2 * (0.4 * ppw * h) ** 2))
        elif self.medium == "sphere":  # plane wave on a sound-soft sphere in c in [0.7, 1.3]
            p = uni(0, 6.28, 3)
            self.c = 1.0 + 0.3 * torch.sin(2 * math.pi * xs[0] + p[0]) * torch.sin(2 * math.pi * xs[1] + p[1]) \
                * torch.sin(2 * math.pi * xs[2] + p[2])
            ppw, c_min, self.dt = 10.0, 0.7, 0.4 * h
            self.mask = (r2 <= (0.1 * min(self.ext)) ** 2).to(torch.uint8)
        else:  # layered: c = 1 / 1.5 / 2 along z, four point sources
            z = xs[-1] / self.ext[-1]
            self.c = torch.where(z < 1 / 3, 1.0, torch.where(z < 2 / 3, 1.5, 2.0)) * one
            ppw, c_min, self.dt = 12.8, 1.0, 0.9 * h / (2.0 * 2.0)
            self.f = 0.0 * one
            for _ in range(4):
                pos = [e * u for e, u in zip(self.ext, uni(0.2, 0.8, self.d))]
                self.f += torch.exp(-sum((x - q) ** 2 for x, q in zip(xs, pos)) / (2 * (0.02 * max(self.ext)) ** 2))
        self.c = self.c.contiguous()
        self.omega = 2 * math.pi * c_min / (ppw * h)
        self.N = max(2, math.ceil(2 * math.pi / self.omega / self.dt - 1e-9))
        if self.f is not None:
            a = uni(0.5, 1.5, 2)
            self.f = torch.complex(a[0] * self.f, 0.0 * self.f)
        else:  # boundary datum of an incident plane wave
            k, dirn = self.omega, uni(-1, 1, self.d)
            nrm = math.sqrt(sum(q * q for q in dirn))
            dirn = [q / nrm for q in dirn]
            ph = k * sum(q * x for q, x in zip(dirn, xs))
            uin = torch.complex(torch.cos(ph), torch.sin(ph)) * one
            acc, cnt = torch.zeros_like(uin), torch.zeros_like(one)
            for a in range(self.d):
                for side in (0, 1):
                    sl = [slice(None)] * self.d
                    sl[self.d - 1 - a] = 0 if side == 0 else n[a]
                    sl = tuple(sl)
                    acc[sl] += 1j * k * ((1.0 if side else -1.0) * dirn[a] - 1.0) * uin[sl]
                    cnt[sl] += 1.0
            self.g = acc / torch.clamp(cnt, min=1.0)
        self.xs, self.one, self.uni = xs, one, uni

    def field(self, scale=1.0):
        """A superposition of plane waves at the problem's wavenumber, 0 on the obstacle."""
        y = torch.zeros(self.shape, device=DEV, dtype=F64)
        for _ in range(5):
            dirn = self.uni(-1, 1, self.d)
            nrm = math.sqrt(sum(q * q for q in dirn)) or 1.0
            y += self.uni(0.3, 1.0)[0] * torch.cos(sum(self.omega * q / nrm * x for q, x in zip(dirn, self.xs))
                                                   + self.uni(0, 6.28)[0])
        if self.mask is not None:
            y = y * (1 - self.mask.to(F64))
        return scale * y

    def inputs(self, op):
        if op in ("wave", "adjoint"):
            # the adjoint takes dual vectors (z = E e): W-weighted amplitudes
            s = 1.0 if op == "wave" else self.h ** self.d
            return self.field(s), self.field(s * (self.omega if op == "wave" else 1.0))
        if op == "riesz":
            return (self.field(self.h ** (self.d - 2)),)
        if op in ("fo_wave", "fo_adjoint"):
            s = 1.0 if op == "fo_wave" else self.h ** self.d
            return (torch.stack([self.field(s * self.omega) for _ in range(self.d + 1)]).reshape(-1),)
        return ()

    def solver(self, case, **kw):
        flags = 0
        if case["op"] in ("fo_wave", "fo_adjoint"):
            flags |= cmcg.FLAG_FIRST_ORDER
        if case.get("vcycle") or case["op"] == "engine":
            flags |= cmcg.FLAG_INEXACT_RIESZ
        if case.get("vcycle") and self.d == 3:
            flags |= cmcg.FLAG_L2_KAPPA
        return cmcg.Solver(self.n, self.h, self.c, self.omega, self.faces, mask=self.mask, order=self.order,
                           precision=PREC[case["prec"]], dt=self.dt, flags=flags, max_iter=case.get("iters", 0),
                           runup_periods=case.get("runup", 0), **kw)


def _engine_cases(case):
    """The uneven members of an engine case, every odd size among them."""
    out = []
    for i in range(case["slots"]):
        m = max(96, int(case["nx"] * (0.4 + 0.6 * ((i * 5 + 3) % 7) / 6.0)) + i)
        out.append(dict(case, nx=m, ny=m))
    return out


# ---- one pass ----------------------------------------------------------------------------------
def prepare(case, seed):
    if case["op"] == "engine":
        eng = cmcg.Engine(max_slots=case["slots"])
        members = []
        for i, m in enumerate(_engine_cases(case)):
            p = _Problem(m, seed, salt=17 * i)
            members.append((p.solver(m, stream=eng.stream), p.f))
        return {"op": "engine", "engine": eng, "members": members}
    p = _Problem(case, seed)
    return {"op": case["op"], "solver": p.solver(case), "in": p.inputs(case["op"]), "f": p.f, "g": p.g}


def run(state):
    op = state["op"]
    if op == "engine":
        eng = state["engine"]
        slots = [eng.submit(s, f=f, tol=1e-10) for s, f in state["members"]]
        done = eng.run_all()
        return [done[k][0] for k in slots]
    s, x = state["solver"], state["in"]
    if op == "wave":
        return s.wave_period(x[0], x[1], state["f"], state["g"])
    if op == "adjoint":
        return s.adjoint_period(x[0], x[1])
    if op == "riesz":
        return s.riesz(x[0])[0]
    if op == "fo_wave":
        return s.fo_period(x[0], state["f"], state["g"])
    if op == "fo_adjoint":
        return s.fo_adjoint_period(x[0])
    return s.solve(state["f"], state["g"], tol=1e-10)[0]


# ---- the work of one pass ----------------------------------------------------------------------
def work(case):
    if case["op"] == "engine":
        parts = [work(dict(m, op="solve", vcycle=True)) for m in _engine_cases(case)]
        return {k: sum(w[k] for w in parts) for k in ("bytes", "flops")}
    d = 3 if case["nz"] else 2
    nodes = (case["nx"] + 1) * (case["ny"] + 1) * (case["nz"] + 1)
    N = {"gauss": 32, "square": 32, "sphere": 36, "layered": 57}.get(case["medium"])
    if N is None:  # random medium
        ppw = 8.0 + 12.0 * (((case["nx"] + case["ny"] + case["nz"]) * 7919) % 1000) / 1000.0
        N = math.ceil(ppw * 2.0 * math.sqrt(d) / 0.9 / (math.sqrt(0.75) if case["order"] == 4 else 1.0))
    # one node update: neighbour sums, 2 y - k L - y_prev (second-order form); link and velocity
    # updates (first-order form)
    upd = {2: 2 * d + 4, 4: 4 * d + 7}[case["order"]]
    esize = 4 if case["prec"] == "fp32" else 8
    src = 16 * nodes
    if case["op"] == "wave":
        return {"bytes": 32 * nodes + src + esize * nodes, "flops": N * upd * nodes}
    if case["op"] == "adjoint":
        return {"bytes": 32 * nodes + 2 * esize * nodes, "flops": N * upd * nodes}
    if case["op"] in ("fo_wave", "fo_adjoint"):
        return {"bytes": 16 * (d + 1) * nodes + esize * nodes + (src if case["op"] == "fo_wave" else 0),
                "flops": N * (5 * d + 5) * nodes}
    if case["op"] == "riesz":
        return {"bytes": 16 * nodes + nodes, "flops": 10 * (2 * d + 20) * nodes}
    grads = case["iters"] + 1
    periods = 2 * grads + case.get("runup", 0) * 1.0
    # per gradient the iterate, residual, direction and gradient pairs are read or written once
    return {"bytes": src + 16 * nodes + grads * 8 * 8 * nodes, "flops": periods * N * upd * nodes}


# ---- the same in plain torch, 64-bit --------------------------------------------------------------
class _Plain:
    """Mass-lumped vertex-centred finite differences and leapfrog, FP64 torch."""

    def __init__(self, p):
        self.p, d = p, p.d
        self.act = p.one if p.mask is None else 1.0 - p.mask.to(F64)
        self.N = p.N
        self.T = 2 * math.pi / p.omega
        self.dt = self.T / p.N
        self.kap = (p.c * self.dt / p.h) ** 2 * self.act
        nb, w = torch.zeros_like(p.one), p.one * p.h ** d
        for a in range(d):
            for side in (0, 1):
                sl = [slice(None)] * d
                sl[d - 1 - a] = 0 if side == 0 else p.n[a]
                nb[tuple(sl)] += 1.0
                w[tuple(sl)] *= 0.5
        self.nb, self.W = nb, w
        self.M = w / p.c ** 2 * self.act
        self.beta = nb * torch.sqrt(self.kap)
        self.S = None
        amp = 0.0
        if p.f is not None:
            amp = amp + p.f
        if p.g is not None:
            amp = amp + (2.0 / p.h) * nb * p.g
        self.S = self.kap * p.h ** 2 * amp

    def _at(self, y, axis, off):
        m = y.shape[axis]
        i = torch.arange(m, device=DEV) + off
        i = torch.where(i < 0, -i, i)
        i = torch.where(i > m - 1, 2 * (m - 1) - i, i)
        return y.index_select(axis, i)

    def lap(self, y):
        out = torch.zeros_like(y)
        for ax in range(self.p.d):
            near = self._at(y, ax, -1) + self._at(y, ax, 1)
            if self.p.order == 2:
                out += 2.0 * y - near
            else:
                out += 2.5 * y - (4.0 / 3.0) * near + (self._at(y, ax, -2) + self._at(y, ax, 2)) / 12.0
        return out

    def force(self, n):
        th = self.p.omega * n * self.dt
        return self.S.real * math.cos(th) + self.S.imag * math.sin(th)

    def period(self, y0, v0, src=True):
        b, k, dt = self.beta, self.kap, self.dt
        y0, v0 = y0 * self.act, v0 * self.act
        f = (lambda n: self.force(n)) if src else (lambda n: 0.0)
        prev = y0
        cur = (y0 + dt * (1 - b) * v0 + 0.5 * (f(0) - k * self.lap(y0))) * self.act
        for n in range(1, self.N):
            prev, cur = cur, ((2 * cur - (1 - b) * prev - k * self.lap(cur) + f(n)) / (1 + b)) * self.act
        vT = ((cur - prev) / dt + (f(self.N) - k * self.lap(cur)) / (2 * dt)) / (1 + b) * self.act
        return cur, vT

    def K(self, y):
        return self.W / self.p.h ** 2 * self.lap(y * self.act) * self.act

    def adjoint(self, a, b):
        dt, M = self.dt, self.M
        live = self.act > 0

        def div(x, y):
            return torch.where(live, x / torch.where(live, y, 1.0), 0.0)

        D, C = M * (1 + self.beta), M * (1 - self.beta)
        t = div(b * self.act, D)
        hi = a * self.act + M * t / dt - (dt / 2) * self.K(t)
        lo = -M * t / dt
        for _ in range(self.N - 1):
            u = div(hi, D)
            hi, lo = lo + 2 * M * u - dt * dt * self.K(u), -C * u
        s = div(hi, M)
        return (lo + hi - (dt * dt / 2) * self.K(s)) * self.act, dt * M * (1 - self.beta) * s * self.act

    def riesz(self, rhs):
        vol = math.prod(self.p.ext)
        b = rhs * self.act
        if self.p.mask is None:
            b = b - b.sum() / vol * self.W
        dg = 1.0 / (2 * self.p.d * self.W / self.p.h ** 2)
        x, r = torch.zeros_like(b), b.clone()
        z = dg * r
        q, rz, stop = z.clone(), (r * z).sum(), float((b * b).sum()) * 1e-28
        for it in range(6000):
            Kq = self.K(q)
            al = rz / (q * Kq).sum()
            x += al * q
            r -= al * Kq
            z = dg * r
            new = (r * z).sum()
            if it % 20 == 19 and float((r * r).sum()) <= stop:
                break
            q = z + new / rz * q
            rz = new
        return x if self.p.mask is not None else x - (self.W * x).sum() / vol

    def gradient(self, w0, w1, src):
        y, v = self.period(w0, w1, src)
        z0, z1 = self.K(y - w0), self.M * (v - w1)
        q0, q1 = self.adjoint(z0, z1)
        return q0 - z0, q1 - z1

    def solve(self, iters):
        live = self.act > 0
        zero = torch.zeros_like(self.W)
        w0, w1 = zero, zero

        def rep(g):
            return self.riesz(g[0]), torch.where(live, g[1] / torch.where(live, self.M, 1.0), 0.0)

        g = self.gradient(w0, w1, True)
        r, rh = rep(g), g
        d = r
        gam = (r[0] * rh[0] + r[1] * rh[1]).sum()
        for _ in range(iters):
            g = self.gradient(d[0], d[1], False)
            gt = rep(g)
            al = gam / (g[0] * d[0] + g[1] * d[1]).sum()
            w0, w1 = w0 - al * d[0], w1 - al * d[1]
            r = (r[0] - al * gt[0], r[1] - al * gt[1])
            rh = (rh[0] - al * g[0], rh[1] - al * g[1])
            new = (r[0] * rh[0] + r[1] * rh[1]).sum()
            d = (r[0] + new / gam * d[0], r[1] + new / gam * d[1])
            gam = new
        om = self.p.omega
        wt, wh = 2 / self.dt * math.sin(om * self.dt / 2), math.sin(om * self.dt) / self.dt
        u = torch.complex(w0, w1 / wh)
        if self.p.mask is None:
            B = 2 * self.beta * self.M / self.dt
            F = torch.where(live, self.S * self.M / self.dt ** 2, 0.0)
            lam = (F.sum() + wt ** 2 * (self.M * u).sum() + 1j * wh * (B * u).sum()) / (wt ** 2 * self.M.sum()
                                                                                     + 1j * wh * B.sum())
            u = (u - lam) * self.act
        return u

    def _end(self, a):
        m = self.p.n[a] + 1
        w = torch.ones(m, device=DEV, dtype=F64)
        w[0] = w[-1] = 0.5
        return w.reshape([-1 if b == self.p.d - 1 - a else 1 for b in range(self.p.d)])

    def fo_period(self, s0, sgn=1.0, src=True):
        """Staggered leapfrog: links p_a (forward differences), then velocities."""
        p, d, h, dt = self.p, self.p.d, self.p.h, self.dt
        s = s0.reshape((d + 1,) + p.shape)
        link = []
        for a in range(d):
            m = torch.ones(p.n[a] + 1, device=DEV, dtype=F64)
            m[-1] = 0.0
            link.append(m.reshape([-1 if b == d - 1 - a else 1 for b in range(d)]))
        P = [s[a] * link[a] for a in range(d)]
        v = s[d] * self.act
        for n in range(self.N):
            div = torch.zeros_like(v)
            for a in range(d):
                ax = d - 1 - a
                P[a] = (P[a] + sgn * dt / h * (torch.roll(v, -1, ax) - v)) * link[a]
                div += (torch.roll(P[a], 1, ax) - P[a]) / self._end(a)
            rhs = (1 - self.beta) * v - sgn * h / dt * self.kap * div
            if src:
                rhs = rhs + self.force(n + 0.5) / dt
            v = rhs / (1 + self.beta) * self.act
        return torch.stack(P + [v]).reshape(-1)

    def fo_adjoint(self, y):
        p, d = self.p, self.p.d
        s = y.reshape((d + 1,) + p.shape)
        live = self.act > 0
        wl = []
        for a in range(d):
            w = torch.full(p.shape, p.h ** d, device=DEV, dtype=F64)
            for b in range(d):
                if b != a:
                    w = w * self._end(b)
            m = torch.ones(p.n[a] + 1, device=DEV, dtype=F64)
            m[-1] = 0.0
            wl.append((w, m.reshape([-1 if b == d - 1 - a else 1 for b in range(d)])))
        D = torch.where(live, self.M * (1 + self.beta), 1.0)
        q = [s[a] / wl[a][0] * wl[a][1] for a in range(d)]
        out = self.fo_period(torch.stack(q + [torch.where(live, s[d] / D, 0.0)]), sgn=-1.0, src=False)
        out = out.reshape((d + 1,) + p.shape)
        return torch.stack([out[a] * wl[a][0] * wl[a][1] for a in range(d)]
                           + [out[d] * self.M * (1 + self.beta)]).reshape(-1)


def exact(case, seed):
    op = case["op"]
    if op == "engine" or case.get("vcycle"):
        return None  # the iterates depend on the V-cycle's own approximation of the Riesz map
    if op == "solve" and case["nz"]:
        return None  # unpreconditioned Riesz solves in 3D take too long here
    if op == "solve" and max(case["nx"], case["ny"]) > 160:
        return None
    p = _Problem(case, seed)
    x, q = p.inputs(op), _Plain(p)
    if op == "wave":
        return q.period(x[0], x[1])
    if op == "adjoint":
        return q.adjoint(x[0], x[1])
    if op == "riesz":
        return q.riesz(x[0])
    if op == "fo_wave":
        return q.fo_period(x[0])
    if op == "fo_adjoint":
        return q.fo_adjoint(x[0])
    return q.solve(case["iters"])
