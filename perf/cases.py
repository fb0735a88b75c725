"""The calls this framework is used for, as cases that can be timed.

A case is one call sequence of a user's program on one grid: a residual, an application of the
preconditioner, smoothing steps, FAS cycles, a steady solve, a physical step of a pitching airfoil,
a cycle of a batch of cases, an adjoint.  ``listed()`` names those of the repository's own
workloads (64x16 ... 1024x256 cells, Euler to thin-layer RANS, FP64 and mixed precision) and some of
odd size; ``draw()`` gives more of the same ranges.  ``prepare`` makes the grid, the seeded initial
state and the solver context a program keeps; ``run`` makes the calls; ``exact`` evaluates the same
equations in plain torch and numpy, in 64 bits.
"""
import ctypes
import math

import numpy as np
import torch

import paper_1710_04875_gb300 as P

GAM = 1.4
PR, PRT, S_COARSE, ETA, D_CUT, RAMP, RAMP_CYCLES = 0.75, 0.9, 0.25, 0.8, 0.5, 20.0, 2
AMP, XC, YC = math.radians(2.0), 0.25, 0.0   # pitching motion: amplitude, axis
OMEGA, STEPS = 0.4, 64                        # reduced frequency 0.2, steps per period
ADJ_ITERS = 10


# ------------------------------------------------------------------------------------------ the cases
def _case(name, kind, flow, ni, nj, levels, precision, **kw):
    c = dict(name=name, kind=kind, flow=flow, ni=ni, nj=nj, levels=levels, precision=precision,
             n_wake=kw.pop("n_wake", ni // 8), scheme="AW3", gamma=1, cfl=100.0, mach=0.75, re=6.5e6, count=1)
    c.update(kw)
    return c


def listed():
    return [
        # the smallest call: one residual of a coarse Euler grid (a caller driving its own iteration)
        _case("residual_64x16", "residual", "euler", 64, 16, 1, "fp64", mach=0.8),
        # the preconditioner alone, on a ragged laminar grid, as a Krylov method would call it
        _case("precond_150x43_laminar", "precond", "laminar", 150, 43, 1, "fp64", mach=0.5, re=5e4, n_wake=18),
        # smoothing steps of a 5-stage W method in mixed precision, no grid hierarchy, odd sizes
        _case("smooth_330x90_aw51_mixed", "smooth", "rans", 330, 90, 1, "mixed", scheme="AW51", n_wake=41, count=2),
        # a short steady solve of a small Euler case: ten V-cycles, a norm read after each
        _case("solve_64x16_euler", "cycle", "euler", 64, 16, 2, "fp64", mach=0.8, cfl=1e4, count=10),
        # the steady Euler workload: 128x32, 3-level V-cycles at the robust pseudo CFL
        _case("cycle_128x32_euler", "cycle", "euler", 128, 32, 3, "fp64", mach=0.8, cfl=1e4, count=3),
        # the steady RANS workload: 256x64, 4-level W-cycles, both precisions
        _case("cycle_256x64_rans", "cycle", "rans", 256, 64, 4, "fp64", gamma=2, mach=0.5, re=1e7, count=3),
        _case("cycle_256x64_rans_mixed", "cycle", "rans", 256, 64, 4, "mixed", gamma=2, mach=0.5, re=1e7, count=3),
        # one physical step of the pitching RANS workload (512x128), three pseudo-time W-cycles
        _case("pitch_512x128_rans_mixed", "pitch", "rans", 512, 128, 4, "mixed", gamma=2, mach=0.8, re=1e6, count=3),
        # the largest workload and the benchmark's headline: 1024x256, one 5-level W-cycle, both precisions
        _case("cycle_1024x256_rans", "cycle", "rans", 1024, 256, 5, "fp64", gamma=2),
        _case("cycle_1024x256_rans_mixed", "cycle", "rans", 1024, 256, 5, "mixed", gamma=2),
        # a cycle of sixteen uneven Euler cases advanced together (a parameter sweep)
        _case("batch16_euler_mixed", "batch", "euler", 512, 128, 4, "mixed", count=16),
        # the adjoint of the RANS workload: Jacobians, a transposed product, ten Krylov iterations
        _case("adjoint_256x64_rans", "adjoint", "rans", 256, 64, 4, "fp64", gamma=2, mach=0.5, re=1e7),
    ]


def draw(rng):
    kind = rng.choice(["residual", "precond", "smooth", "cycle", "cycle", "cycle", "pitch", "batch", "adjoint"])
    flow = "rans" if kind == "pitch" else "euler" if kind == "batch" else rng.choice(["euler", "laminar", "rans", "rans"])
    low, top = dict(pitch=(128, 512), batch=(96, 512), adjoint=(48, 224)).get(kind, (48, 1000))
    ni = int(math.exp(rng.uniform(math.log(low), math.log(top))))
    nj = max(10, min(256, int(ni * rng.uniform(0.18, 0.34))))
    levels = 1
    if kind in ("cycle", "pitch", "batch", "adjoint"):   # whole cycles: sizes that agglomerate
        levels = rng.randint(3, 4) if kind == "pitch" else rng.randint(1, 5)
        while levels > 1 and nj >> (levels - 1) < 8:
            levels -= 1
    f = 1 << (levels - 1)
    ni, nj = max(2 * f, ni // (2 * f) * 2 * f), max(8, nj // f * f)
    n_wake = max(f, round(ni / rng.uniform(7.0, 12.0) / f) * f)
    scheme = rng.choice(["AW3", "AW51", "ARK3J"]) if kind == "smooth" else "AW3"
    count = dict(smooth=rng.randint(1, 3), cycle=rng.randint(1, 3) if ni < 600 else 1, pitch=rng.randint(1, 3),
                 batch=rng.randint(4, 14)).get(kind, 1)
    return dict(kind=kind, flow=flow, ni=ni, nj=nj, levels=levels, n_wake=n_wake,
                precision="fp64" if kind == "adjoint" else rng.choice(["fp64", "mixed"]), scheme=scheme,
                gamma=1 if levels == 1 else rng.choice([1, 2]), cfl=1.0 if scheme == "ARK3J" else 100.0,
                mach=round(rng.uniform(0.5, 0.8), 3), re=round(10 ** rng.uniform(4.3, 5.0)) if flow == "laminar" else
                round(10 ** rng.uniform(6.0, 7.0)), count=count)


def _members(case):
    """The cases of a batch: sizes spread over 128 ... ni in steps of 32, other flow conditions each."""
    if case["kind"] != "batch":
        return [case]
    out, n = [], case["count"]
    for k in range(n):
        ni = max(64, int(case["ni"] * (0.25 + 0.75 * ((5 * k) % n) / max(1, n - 1))) // 32 * 32)
        nj = ni // 4
        lev = case["levels"]
        while lev > 1 and (nj >> (lev - 1) < 8 or nj % (1 << (lev - 1))):
            lev -= 1
        f = max(8, 1 << (lev - 1))
        out.append(dict(case, ni=ni, nj=nj, levels=lev, n_wake=f * max(1, round(ni / 64)),
                        mach=0.5 + 0.3 * ((3 * k) % n) / n))
    return out


def _alpha(case):
    return 0.0 if case["flow"] == "rans" and case["kind"] != "adjoint" else 1.25


# ------------------------------------------------------------------------------------------ inputs
def _ratio(first, n, length):
    lo, hi = 1.0 + 1e-12, 3.0
    for _ in range(100):
        mid = 0.5 * (lo + hi)
        lo, hi = (mid, hi) if first * (mid ** n - 1.0) / (mid - 1.0) < length else (lo, mid)
    return 0.5 * (lo + hi)


class Grid:
    """C-grid around a closed NACA 0010 section: straight lines leave the wall and the wake along
    smoothly turning directions; half of the cells of a line lie in the boundary layer."""

    def __init__(self, ni, nj, n_wake, first):
        self.ni, self.nj, self.n_wake = ni, nj, n_wake
        side = ni // 2 - n_wake
        k = np.arange(side + 1)
        xu = 0.5 * (1.0 - np.cos(np.pi * k / side))
        yu = 0.5 * (0.2969 * np.sqrt(xu) - 0.1260 * xu - 0.3516 * xu ** 2 + 0.2843 * xu ** 3 - 0.1036 * xu ** 4)
        yu[0] = yu[-1] = 0.0
        h0 = xu[-1] - xu[-2]
        q = np.arange(1, n_wake + 1)
        wake = 10.0 * q / n_wake if h0 * n_wake >= 10.0 else None
        if wake is None:
            r = _ratio(h0, n_wake, 10.0)
            wake = h0 * (r ** q - 1.0) / (r - 1.0)
        x0 = np.concatenate([xu, 1.0 + wake])                      # leading edge ... outflow, upper side
        y0 = np.concatenate([yu, np.zeros(n_wake)])
        te = math.atan(0.5 * (0.2969 / 2 - 0.1260 - 0.7032 + 0.8529 - 0.4144))  # surface angle at the trailing edge
        tx, ty = np.gradient(x0[:side + 1]), np.gradient(y0[:side + 1])
        ang = np.arctan2(tx, -ty)                                   # direction of the outward line
        ang[0], ang[side] = math.pi, 0.5 * math.pi + te
        lean = np.linspace(ang[side], math.pi / 2 - max(0.3, -te + 0.05), n_wake + 1)[1:]
        ang = np.concatenate([ang, lean])
        n1 = nj // 2
        rb = _ratio(first, n1, max(0.05, 2.0 * first * n1))
        sp = first * rb ** np.arange(n1)
        r2 = _ratio(sp[-1], nj - n1 + 1, 20.0 - sp.sum() + sp[-1])
        sp = np.concatenate([sp, sp[-1] * r2 ** np.arange(1, nj - n1 + 1)])
        d = np.concatenate([[0.0], np.cumsum(sp)])[:, None]
        xu, yu = x0 + d * np.cos(ang), y0 + d * np.sin(ang)
        xu[:, 0], yu[:, 0] = -d[:, 0], 0.0
        self.x = np.ascontiguousarray(np.concatenate([xu[:, :0:-1], xu], axis=1))
        self.y = np.ascontiguousarray(np.concatenate([-yu[:, :0:-1], yu], axis=1))

    def coords(self):
        return self.x.ravel(), self.y.ravel()


def _grid(case):
    return Grid(case["ni"], case["nj"], case["n_wake"], dict(euler=2e-3, laminar=5e-4, rans=1e-5)[case["flow"]])


def _free_stream(case):
    al, p = math.radians(_alpha(case)), 1.0 / (GAM * case["mach"] ** 2)
    return np.array([1.0, math.cos(al), math.sin(al), p / (GAM - 1.0) + 0.5])


def _state(case, g, rng):
    """A flow on its way to the steady state: the free stream, slowed to rest through a layer at the
    wall in viscous flow, with smooth disturbances of density, velocity and pressure."""
    ni, nj = g.ni, g.nj
    cx = 0.25 * (g.x[1:, 1:] + g.x[:-1, 1:] + g.x[1:, :-1] + g.x[:-1, :-1])
    cy = 0.25 * (g.y[1:, 1:] + g.y[:-1, 1:] + g.y[1:, :-1] + g.y[:-1, :-1])
    xw, yw = 0.5 * (g.x[0, 1:] + g.x[0, :-1]), 0.5 * (g.y[0, 1:] + g.y[0, :-1])
    dist = np.hypot(cx - xw, cy - yw)
    s, t = np.arange(ni)[None, :] / ni, np.arange(nj)[:, None] / nj

    def wave():
        out = np.zeros((nj, ni))
        for _ in range(3):
            a, b, c = rng.integers(1, 5), rng.integers(1, 4), rng.uniform(0.0, 2.0 * np.pi)
            out += rng.uniform(0.3, 1.0) * np.sin(2.0 * np.pi * a * s + c) * np.cos(np.pi * b * t)
        return out * (1.0 - t) ** 2

    w = _free_stream(case)
    rho, u, v = 1.0 + 0.004 * wave(), w[1] + 0.004 * wave(), w[2] + 0.004 * wave()
    p = (1.0 + 0.004 * wave()) / (GAM * case["mach"] ** 2)
    if case["flow"] != "euler":
        layer = np.tanh(dist / (0.004 if case["flow"] == "rans" else 0.02))
        wall = (np.arange(ni) >= g.n_wake) & (np.arange(ni) < ni - g.n_wake)
        f = np.where(wall[None, :], layer, 1.0 - (1.0 - layer) * np.exp(-2.0 * np.maximum(xw - 1.0, 0.0))[None, :])
        u, v = u * f, v * f
    return np.ascontiguousarray(np.stack([rho, rho * u, rho * v, p / (GAM - 1.0) + 0.5 * rho * (u * u + v * v)]))


def _inputs(case, seed):
    """Per member: case, grid, initial state, and a vector for what applies an operator to one."""
    out = []
    for k, m in enumerate(_members(case)):
        rng = np.random.default_rng([seed, k])
        g = _grid(m)
        u = _state(m, g, rng)
        v = rng.standard_normal(u.shape)
        out.append((m, g, u, 1e-3 * v if case["kind"] == "precond" else v))
    return out


def _params(c):
    return P.default_params(scheme=c["scheme"], nlevels=c["levels"], gamma_cycle=c["gamma"],
                            viscous=int(c["flow"] != "euler"), turb=int(c["flow"] == "rans"),
                            sensor=int(c["flow"] != "euler"), mach=c["mach"], alpha_deg=_alpha(c), re=c["re"],
                            cfl=c["cfl"], precision=c["precision"])


class State:
    pass


def prepare(case, seed):
    st = State()
    st.case, st.kind, st.count = case, case["kind"], case["count"]
    members = _inputs(case, seed)
    st.stream = torch.cuda.Stream()      # cycles are replayed as CUDA graphs on a stream of one's own
    st.lib = P.fasw.library()
    st.norm = ctypes.c_double()
    st.step = 0
    st.u0 = [torch.from_numpy(u).cuda() for _, _, u, _ in members]
    st.v = torch.from_numpy(members[0][3]).cuda() if st.kind in ("precond", "adjoint") else None
    st.out = [torch.empty_like(u) for u in st.u0]
    st.more = [torch.empty_like(st.u0[0]) for _ in range(2)] if st.kind in ("residual", "adjoint") else None
    if st.kind == "batch":
        st.batch = P.fasw.Batch([g for _, g, _, _ in members], [_params(m) for m, _, _, _ in members],
                                stream=st.stream.cuda_stream)
        st.handles = [(st.lib.fasw_batch_case(st.batch.h, k), m["levels"] - 1) for k, (m, _, _, _) in enumerate(members)]
    else:
        m, g, _, _ = members[0]
        st.solver = P.Solver(g, _params(m), stream=st.stream.cuda_stream)
        st.solver.set_state(st.u0[0])
        st.handles = [(st.solver.h, m["levels"] - 1)]
    torch.cuda.synchronize()
    return st


def _ok(code):
    if code != 0:
        raise RuntimeError(f"call failed with code {code}")


# ------------------------------------------------------------------------------------------ one pass
def run(st):
    kind, lib = st.kind, st.lib
    if kind == "batch":
        for (h, l), u in zip(st.handles, st.u0):
            _ok(lib.fasw_set_state(h, l, u.data_ptr(), 1))
        norms = st.batch.cycle(RAMP_CYCLES)
        for (h, l), out in zip(st.handles, st.out):
            _ok(lib.fasw_get_state(h, l, out.data_ptr(), 1))
        return [norms] + st.out
    s, (h, l), out = st.solver, st.handles[0], st.out[0]
    if kind == "residual":
        _ok(lib.fasw_residual(h, l, out.data_ptr(), st.more[0].data_ptr(), st.more[1].data_ptr(), 1,
                              ctypes.byref(st.norm)))
        return [out, st.more[0], st.more[1], st.norm.value]
    if kind == "precond":
        _ok(lib.fasw_precond_apply(h, l, st.case["cfl"], st.v.data_ptr(), out.data_ptr(), 1))
        return [out]
    if kind == "smooth":
        s.set_state(st.u0[0])
        s.smooth(st.count, st.case["cfl"])
        return [s.get_state(out=out)]
    if kind == "cycle":
        s.set_state(st.u0[0])
        first = RAMP_CYCLES if st.count == 1 else 0
        norms = [s.fas_cycle(first + k) for k in range(st.count)]
        return [s.get_state(out=out), np.array(norms)]
    if kind == "pitch":       # each pass is the next physical step of the motion
        st.step += 1
        dt = 2.0 * math.pi / OMEGA / STEPS
        t = OMEGA * dt * st.step
        s.set_motion(-AMP * math.sin(t), -AMP * OMEGA * math.cos(t), XC, YC)
        _, _, norms = s.dual_time_step(dt, 1e-11, st.count)
        return [s.get_state(out=out), norms]
    s.set_state(st.u0[0])     # adjoint: the eddy viscosity of this state, its Jacobians, J^T v, some Krylov steps
    mut = [s.get_mut()] if st.case["flow"] == "rans" else []
    s.adjoint_jacobian()
    jtv = s.adjoint_apply(st.v, transpose=True, out=out)
    lam = s.adjoint_solve(which=1, tol=1e-14, max_iters=ADJ_ITERS)[0]
    return [jtv, lam] + mut


# ------------------------------------------------------------------------------------------ its work
def work(case):
    """Bytes and operations of a pass.  Per cell and evaluation: a residual reads the state, metrics
    and volume and writes F (about 310 operations); a smoothing step builds two faces' Jacobians and
    the factored diagonal (about 480) and, per stage, takes a residual and a forward and backward
    sweep (about 290).  Everything between could stay on the chip: the bytes are the state in and out
    per level visit and the grid once."""
    stages = 5 if case["scheme"].startswith("AW5") else 3
    nbytes = flops = 0.0
    for m in _members(case):
        n = m["ni"] * m["nj"]
        grid = 8.0 * (2 * n + 2 * n + n)
        kind = case["kind"]
        if kind == "residual":
            b, f = grid + 32.0 * 4 * n + 8.0, 400.0 * n
        elif kind == "precond":
            b, f = grid + 32.0 * 3 * n, (60.0 + 480.0 + 290.0) * n
        elif kind == "adjoint":
            solves = 4.0 / 3.0 if m["levels"] > 1 else 1.0
            per_cycle = 31.0 * 2 * 11 * 16 + stages * (290.0 + 4 * 11 * 32)
            b = grid + 32.0 * 4 * n + (8.0 * n if m["flow"] == "rans" else 0.0)
            f = solves * n * (11 * 16 * 40.0 + ADJ_ITERS * per_cycle)
        else:
            b = f = 0.0
            cycles = 1 if kind == "batch" else m["count"]
            for l in range(m["levels"]):
                cells, visits = n / 4.0 ** l, float(m["gamma"]) ** l * cycles
                b += visits * cells * 8.0 * (4 + 4 + 5)
                f += visits * cells * (480.0 + stages * (400.0 + 290.0) + (800.0 if m["levels"] > 1 else 0.0))
        nbytes, flops = nbytes + b, flops + f
    return {"bytes": nbytes, "flops": flops}


# ------------------------------------------------------------------- the same in 64 bits, from the equations
class _Level:
    """Metrics of one level, (rows, columns) arrays; vectors have a leading axis of 2."""

    def __init__(self, g=None, fine=None, phi=0.0, rate=0.0):
        if fine is None:
            self.ni, self.nj, self.nw = g.ni, g.nj, g.n_wake
            dx, dy, c, s = g.x - XC, g.y - YC, math.cos(phi), math.sin(phi)
            x, y = (g.x, g.y) if phi == 0.0 else (XC + c * dx - s * dy, YC + s * dx + c * dy)
            self.sx = np.stack([y[1:] - y[:-1], -(x[1:] - x[:-1])])
            self.se = np.stack([-(y[:, 1:] - y[:, :-1]), x[:, 1:] - x[:, :-1]])
            mx, my = 0.5 * (x[1:] + x[:-1]), 0.5 * (y[1:] + y[:-1])
            self.vx = rate * (-(my - YC) * self.sx[0] + (mx - XC) * self.sx[1])
            mx, my = 0.5 * (x[:, 1:] + x[:, :-1]), 0.5 * (y[:, 1:] + y[:, :-1])
            self.ve = rate * (-(my - YC) * self.se[0] + (mx - XC) * self.se[1])
            self.wall = rate * np.stack([-(my[0] - YC), mx[0] - XC])
            d1x, d1y = x[1:, 1:] - x[:-1, :-1], y[1:, 1:] - y[:-1, :-1]
            d2x, d2y = x[1:, :-1] - x[:-1, 1:], y[1:, :-1] - y[:-1, 1:]
            self.vol = 0.5 * (d1x * d2y - d1y * d2x)
            cx = 0.25 * (x[1:, 1:] + x[:-1, 1:] + x[1:, :-1] + x[:-1, :-1])
            cy = 0.25 * (y[1:, 1:] + y[:-1, 1:] + y[1:, :-1] + y[:-1, :-1])
            self.dist = np.hypot(cx - mx[0], cy - my[0])
        else:
            self.ni, self.nj, self.nw = fine.ni // 2, fine.nj // 2, fine.nw // 2
            self.sx = fine.sx[:, 0::2, 0::2] + fine.sx[:, 1::2, 0::2]
            self.se = fine.se[:, 0::2, 0::2] + fine.se[:, 0::2, 1::2]
            self.vx = fine.vx[0::2, 0::2] + fine.vx[1::2, 0::2]
            self.ve = fine.ve[0::2, 0::2] + fine.ve[0::2, 1::2]
            self.wall = 0.5 * (fine.wall[:, 0::2] + fine.wall[:, 1::2])
            self.vol = self.sum4(fine.vol)
        i = np.arange(self.ni)
        self.cut = (i < self.nw) | (i >= self.ni - self.nw)
        for k in ("sx", "se", "vx", "ve", "wall", "vol"):
            setattr(self, "t_" + k, torch.from_numpy(np.ascontiguousarray(getattr(self, k))))
        self.t_cut = torch.from_numpy(self.cut)

    @staticmethod
    def sum4(a):
        return (a[..., 0::2, 0::2] + a[..., 0::2, 1::2]) + (a[..., 1::2, 0::2] + a[..., 1::2, 1::2])


class _Exact:
    """The discretization and the FAS cycle of arXiv 1710.04875 (JST flux, thin-layer stresses,
    Baldwin-Lomax, flux-vector-split block SGS), 64 bits, vectorized over cells and hyperplanes."""

    ALPHA = dict(AW3=(0.1481, 0.4, 1.0), AW51=(0.0533, 0.1263, 0.2375, 0.4414, 1.0))
    BETA = dict(AW3=(1.0, 0.5, 0.5), AW51=(1.0, 0.0, 0.56, 0.0, 0.44))

    def __init__(self, case, grid, phi=0.0, rate=0.0):
        self.c = case
        self.viscous, self.turb = case["flow"] != "euler", case["flow"] == "rans"
        self.winf = _free_stream(case)
        self.mu = 1.0 / case["re"]
        name = case["scheme"].replace("ARK3J", "AW3")
        self.alpha, self.beta = self.ALPHA[name], self.BETA[name]
        self.aw = case["scheme"].startswith("AW")
        self.lev = [_Level(grid, phi=phi, rate=rate)]
        while len(self.lev) < case["levels"]:
            self.lev.append(_Level(fine=self.lev[-1]))     # 0 is the finest
        self.mut = [np.zeros((L.nj, L.ni)) for L in self.lev]
        self.at, self.src = 0.0, 0.0

    @staticmethod
    def prim(w):
        u, v = w[1] / w[0], w[2] / w[0]
        p = (GAM - 1.0) * (w[3] - 0.5 * (w[1] * u + w[2] * v))
        return w[0], u, v, p

    def far(self, w, n, vb):
        r, u, v, p = self.prim(w)
        a = torch.sqrt(GAM * p / r)
        ri, ui, vi, pi = self.prim(self.winf)
        ai = math.sqrt(GAM * pi / ri)
        vn, vni = u * n[0] + v * n[1], ui * n[0] + vi * n[1]
        rp, rm = vn + 5.0 * a, vni - 5.0 * ai
        vnb, ab = 0.5 * (rp + rm), 0.1 * (rp - rm)
        out = vnb - vb > 0.0
        rup, aup = torch.where(out, r, ri + 0 * r), torch.where(out, a, ai + 0 * a)
        ut = torch.where(out, u - vn * n[0], ui - vni * n[0])
        vt = torch.where(out, v - vn * n[1], vi - vni * n[1])
        rho = rup * (ab / aup) ** 5
        ub, vb2 = ut + vnb * n[0], vt + vnb * n[1]
        g = torch.stack([rho, rho * ub, rho * vb2, rho * ab ** 2 / GAM / (GAM - 1.0) + 0.5 * rho * (ub ** 2 + vb2 ** 2)])
        sup = torch.abs(vn - vb) >= a
        up = torch.where(vn - vb > 0.0, w, torch.from_numpy(self.winf)[:, None] + 0 * w)
        return torch.where(sup, up, g)

    def ghosts(self, L, u):
        """(4, nj + 4, ni + 4): two ghost layers on every side."""
        rows = []
        for k in (1, 0):
            w = u[:, k]
            r, a, b, p = self.prim(w)
            n = L.t_se[:, 0] / torch.sqrt((L.t_se[:, 0] ** 2).sum(0))
            if self.viscous:
                ug, vg = 2.0 * L.t_wall[0] - a, 2.0 * L.t_wall[1] - b
            else:
                rn = (a - L.t_wall[0]) * n[0] + (b - L.t_wall[1]) * n[1]
                ug, vg = a - 2.0 * rn * n[0], b - 2.0 * rn * n[1]
            g = torch.stack([r, r * ug, r * vg, p / (GAM - 1.0) + 0.5 * r * (ug * ug + vg * vg)])
            rows.append(torch.where(L.t_cut, w.flip(-1), g)[:, None])
        ln = torch.sqrt((L.t_se[:, -1] ** 2).sum(0))
        top = self.far(u[:, -1], L.t_se[:, -1] / ln, L.t_ve[-1] / ln)[:, None]
        mid = torch.cat([rows[0], rows[1], u, top, top], dim=1)
        l0, l1 = (torch.sqrt((L.t_sx[:, :, k] ** 2).sum(0)) for k in (0, -1))
        left = self.far(u[:, :, 0], -L.t_sx[:, :, 0] / l0, -L.t_vx[:, 0] / l0)
        right = self.far(u[:, :, -1], L.t_sx[:, :, -1] / l1, L.t_vx[:, -1] / l1)
        corner = torch.from_numpy(self.winf)[:, None, None].expand(4, 2, 1)
        left, right = (torch.cat([corner, c[:, :, None], corner], dim=1) for c in (left, right))
        return torch.cat([left, left, mid, right, right], dim=2)

    def radii(self, L, u):
        r, a, b, p = self.prim(u)
        c = torch.sqrt(GAM * p / r)
        out = []
        for S, V in ((0.5 * (L.t_sx[:, :, 1:] + L.t_sx[:, :, :-1]), 0.5 * (L.t_vx[:, 1:] + L.t_vx[:, :-1])),
                     (0.5 * (L.t_se[:, 1:] + L.t_se[:, :-1]), 0.5 * (L.t_ve[1:] + L.t_ve[:-1]))):
            out.append(torch.abs(a * S[0] + b * S[1] - V) + c * torch.sqrt((S ** 2).sum(0)))
        return out

    def residual(self, l, u, mut):
        """F^c and F^v per volume without time and forcing terms; u (4, nj, ni) torch, mut numpy."""
        L, ni, nj = self.lev[l], self.lev[l].ni, self.lev[l].nj
        G = self.ghosts(L, u)
        rx, re = self.radii(L, u)
        tx, te = rx * (1.0 + (re / rx) ** (2.0 / 3.0)), re * (1.0 + (rx / re) ** (2.0 / 3.0))
        tx = torch.cat([tx[:, :1], tx, tx[:, -1:]], dim=1)
        te = torch.cat([torch.where(L.t_cut, te[0].flip(-1), te[0])[None], te, te[-1:]], dim=0)
        r, a, b, p = self.prim(G)
        q = p * r ** -GAM if self.viscous else p
        W = torch.cat([G[:3], (G[3] + p)[None]])
        fc, fd = [], []
        for d in (0, 1):
            if d == 0:
                cut4 = [(slice(2, -2), slice(k, k + ni + 1)) for k in range(4)]
                S, V, rt = L.t_sx, L.t_vx, torch.maximum(tx[:, 1:], tx[:, :-1])
            else:
                cut4 = [(slice(k, k + nj + 1), slice(2, -2)) for k in range(4)]
                S, V, rt = L.t_se, L.t_ve, torch.maximum(te[1:], te[:-1])
            h = 0.0
            for k in (1, 2):
                g, pk = G[(slice(None),) + cut4[k]], p[cut4[k]]
                qn = (g[1] * S[0] + g[2] * S[1]) / g[0]
                h = h + 0.5 * torch.stack([g[0] * qn, g[1] * qn + pk * S[0], g[2] * qn + pk * S[1], (g[3] + pk) * qn])
                h = h - 0.5 * g * V
            w = [W[(slice(None),) + c] for c in cut4]
            d0 = w[2] - w[1]
            if l == 0:
                qs = [q[c] for c in cut4]
                sen = [torch.abs(qs[k + 1] - 2.0 * qs[k] + qs[k - 1]) / (qs[k + 1] + 2.0 * qs[k] + qs[k - 1] + 0.001)
                       for k in (1, 2)]
                e2 = torch.clamp(torch.maximum(*sen), max=0.25) * rt
                e4 = torch.clamp(rt / 32.0 - 2.0 * e2, min=0.0)
                dis = e2 * d0 - e4 * ((w[3] - w[2]) + (w[1] - w[0]) - 2.0 * d0)
            else:
                dis = S_COARSE * rt * d0
            if d == 1 and self.viscous:
                dis = dis + self.viscous_flux(L, G, p, mut)
            fc.append(h)
            fd.append(dis)
        div = [(x[0][:, :, 1:] - x[0][:, :, :-1]) + (x[1][:, 1:] - x[1][:, :-1]) for x in (fc, fd)]
        return div[0] / L.t_vol, -div[1] / L.t_vol

    def face_means(self, L, mut):
        """Volume sums and eddy viscosity at the j-faces."""
        vol = np.concatenate([np.where(L.cut, L.vol[0, ::-1], L.vol[0])[None], L.vol, L.vol[-1:]])
        m = np.concatenate([np.where(L.cut, mut[0, ::-1], -mut[0])[None], mut, mut[-1:]])
        return vol[1:] + vol[:-1], 0.5 * (m[1:] + m[:-1])

    def viscous_flux(self, L, G, p, mut):
        vs, mf = (torch.from_numpy(np.ascontiguousarray(x)) for x in self.face_means(L, mut))
        S = L.t_se
        gl, gr, pl, pr = G[:, 1:-2, 2:-2], G[:, 2:-1, 2:-2], p[1:-2, 2:-2], p[2:-1, 2:-2]
        ul, vl, ur, vr = gl[1] / gl[0], gl[2] / gl[0], gr[1] / gr[0], gr[2] / gr[0]
        hl, hr = 3.5 * pl / gl[0], 3.5 * pr / gr[0]
        k = 2.0 / vs
        gux, guy, gvx, gvy = (ur - ul) * S[0] * k, (ur - ul) * S[1] * k, (vr - vl) * S[0] * k, (vr - vl) * S[1] * k
        me, ke = self.mu + mf, self.mu / PR + mf / PRT
        div = gux + gvy
        xx, yy, xy = me * (2.0 * gux - 2.0 / 3.0 * div), me * (2.0 * gvy - 2.0 / 3.0 * div), me * (guy + gvx)
        fx, fy = xx * S[0] + xy * S[1], xy * S[0] + yy * S[1]
        heat = ke * (hr - hl) * k * (S ** 2).sum(0)
        return torch.stack([0.0 * fx, fx, fy, 0.5 * (ul + ur) * fx + 0.5 * (vl + vr) * fy + heat])

    def eddy(self, u):
        """Baldwin-Lomax on the finest level."""
        L = self.lev[0]
        G = self.ghosts(L, torch.from_numpy(u)).numpy()
        uu, vv, ni, nj = G[1] / G[0], G[2] / G[0], L.ni, L.nj
        cir = 0.0
        c = (slice(2, -2), slice(2, -2))
        for sgn, S, nb in ((1, L.sx[:, :, 1:], (slice(2, -2), slice(3, -1))), (-1, L.sx[:, :, :-1], (slice(2, -2), slice(1, -3))),
                           (1, L.se[:, 1:], (slice(3, -1), slice(2, -2))), (-1, L.se[:, :-1], (slice(1, -3), slice(2, -2)))):
            cir = cir + sgn * (0.5 * (vv[c] + vv[nb]) * S[0] - 0.5 * (uu[c] + uu[nb]) * S[1])
        om, y, rho = np.abs(cir / L.vol), L.dist, u[0]
        sp = np.hypot(u[1] / rho, u[2] / rho)
        utr = np.sqrt(rho[0] * self.mu * om[0])
        damp = np.where(L.cut, 1.0, 1.0 - np.exp(-y * utr * self.c["re"] / 26.0))
        F, js = (y * om * damp), max(1, nj // 2)
        jm = F[:js].argmax(0)
        fm = F[:js].max(0)
        ym = np.where(fm > 0.0, np.take_along_axis(y, jm[None], 0)[0], 0.0)
        ud = np.where(L.cut, sp[:js].max(0) - sp[:js].min(0), sp[:js].max(0))
        fs, ys = np.where(fm > 0.0, fm, 1.0), np.where(ym > 0.0, ym, 1.0)
        fw = np.where(fm > 0.0, np.minimum(ym * fm, 0.25 * ym * ud * ud / fs), 0.0)
        mo = 0.0168 * 1.6 * rho * fw * np.where(ym > 0.0, 1.0 / (1.0 + 5.5 * (0.3 * y / ys) ** 6), 0.0)
        mi = rho * (0.4 * y * damp) ** 2 * om
        outer = np.logical_or.accumulate((mi >= mo) | L.cut, axis=0)
        return np.where(outer, mo, mi)

    def split(self, L, G, mut):
        """|S| A+, |S| A- at the i-faces and j-faces, (rows, columns, 4, 4)."""
        ni, nj = L.ni, L.nj
        out = []
        for d in (0, 1):
            if d == 0:
                w, S, V = 0.5 * (G[:, 2:-2, 1:ni + 2] + G[:, 2:-2, 2:ni + 3]), L.sx, L.vx
            else:
                w, S, V = 0.5 * (G[:, 1:nj + 2, 2:-2] + G[:, 2:nj + 3, 2:-2]), L.se, L.ve
            ln = np.sqrt((S ** 2).sum(0))
            nx, ny = S / ln
            rho, u, v, p = self.prim(w)
            a, H, q2 = np.sqrt(GAM * p / rho), (w[3] + p) / rho, u * u + v * v
            vn = u * nx + v * ny
            vr = vn - V / ln
            r0, r1 = np.stack([1.0 + 0 * u, u, v, H]), np.stack([0 * u, nx, ny, vn])
            dp = (GAM - 1.0) * np.stack([0.5 * q2, -u, -v, 1.0 + 0 * u])
            dv = np.stack([-vn, nx, ny, 0 * u])
            lam = [vr, vr + a, vr - a]
            ad = a * D_CUT
            ab = [np.where(np.abs(x) <= ad, 0.5 * (ad + x * x / ad), np.abs(x)) for x in lam]
            for s in (1.0, -1.0):
                l1, l3, l4 = (0.5 * (x + s * y) for x, y in zip(lam, ab))
                c1, c2 = 0.5 * (l3 + l4) - l1, 0.5 * (l3 - l4)
                g0, g1 = c1 / a ** 2 * dp + c2 / a * dv, c2 / a * dp + c1 * dv
                M = l1 * np.eye(4)[:, :, None, None] + r0[:, None] * g0[None] + r1[:, None] * g1[None]
                M = M * ln
                if d == 1 and self.viscous:
                    vs, mf = self.face_means(L, mut)
                    nu = np.maximum(self.mu + mf, GAM * (self.mu / PR + mf / PRT)) / w[0]
                    M = M + s * (2.0 * nu * ln ** 2 / vs) * np.eye(4)[:, :, None, None]
                out.append(np.ascontiguousarray(M.transpose(2, 3, 0, 1)))
        return out

    def steps_dt(self, L, u, cfl):
        rx, re = self.radii(L, torch.from_numpy(u))
        return cfl * L.vol / (rx + re).numpy()

    def factor(self, l, u, cfl, mut):
        """Pseudo time step and the blocks of P = (D + L) D^-1 (D + U) at the state u."""
        L = self.lev[l]
        dts = self.steps_dt(L, u, cfl)
        G = self.ghosts(L, torch.from_numpy(u)).numpy()
        xp, xm, ep, em = self.split(L, G, mut)
        cf = (ETA * dts / L.vol if self.aw else 1.0 / L.vol)[..., None, None]
        sg = (1.0 + ETA * dts * self.at if self.aw else self.at + 0 * dts)[..., None, None]
        D = sg * np.eye(4) + cf * ((xp[:, 1:] - xm[:, :-1]) + (ep[1:] - em[:-1]))
        Di = np.linalg.inv(D)
        return dts, (Di, cf * xp[:, :-1], cf * ep[:-1], cf * xm[:, 1:], cf * em[1:])

    def sgs(self, L, blocks, r):
        """z = P^-1 r by the forward and backward sweep along the hyperplanes i + j."""
        Di, Aw, As, Ae, An = blocks
        ni, nj, nw = L.ni, L.nj, L.nw
        r = np.ascontiguousarray(r.transpose(1, 2, 0))[..., None]
        y = np.zeros((nj, ni, 4, 1))
        planes = []
        for k in range(ni + nj - 1):
            i = np.arange(max(0, k - nj + 1), min(k, ni - 1) + 1)
            planes.append((k - i, i))
        for j, i in planes:
            t = r[j, i]
            m = i > 0
            t[m] += Aw[j[m], i[m]] @ y[j[m], i[m] - 1]
            m = j > 0
            t[m] += As[j[m], i[m]] @ y[j[m] - 1, i[m]]
            if j[-1] == 0 and i[-1] >= ni - nw:
                t[-1] += As[0, i[-1]] @ y[0, ni - 1 - i[-1]]
            y[j, i] = Di[j, i] @ t
        for j, i in reversed(planes):
            t = np.zeros((len(i), 4, 1))
            m = i < ni - 1
            t[m] += Ae[j[m], i[m]] @ y[j[m], i[m] + 1]
            m = j < nj - 1
            t[m] += An[j[m], i[m]] @ y[j[m] + 1, i[m]]
            if j[-1] == 0 and i[-1] < nw:
                t[-1] -= As[0, i[-1]] @ y[0, ni - 1 - i[-1]]
            y[j, i] -= Di[j, i] @ t
        return y[..., 0].transpose(2, 0, 1)

    def smooth(self, l, u, cfl, s):
        """One smoothing step; returns the state and the density norm of the first residual."""
        dts, blocks = self.factor(l, u, cfl, self.mut[l])
        u0, carry, norm = u, None, None
        for al, be in zip(self.alpha, self.beta):
            Fc, Fv = (x.numpy() for x in self.residual(l, torch.from_numpy(np.ascontiguousarray(u)), self.mut[l]))
            Fc = Fc + self.at * u - s + (self.src if l == 0 else 0.0)
            carry = Fv if carry is None else be * Fv + (1.0 - be) * carry
            norm = math.sqrt(float(np.mean((Fc[0] + Fv[0]) ** 2))) if norm is None else norm
            z = self.sgs(self.lev[l], blocks, (dts if self.aw else 1.0) * (Fc + carry))
            u = np.ascontiguousarray(u0 - al * (1.0 if self.aw else dts) * z)
        return u, norm

    def fas(self, l, u, cfl, s):
        u, norm = self.smooth(l, u, cfl, s)
        if l == len(self.lev) - 1:
            return u, norm
        F, C = self.lev[l], self.lev[l + 1]
        Fc, Fv = (x.numpy() for x in self.residual(l, torch.from_numpy(u), self.mut[l]))
        r = s - (Fc + Fv + self.at * u + (self.src if l == 0 else 0.0))
        uc, rc = C.sum4(F.vol * u) / C.vol, C.sum4(F.vol * r) / C.vol
        if self.turb:
            self.mut[l + 1] = C.sum4(F.vol * self.mut[l]) / C.vol
        Fc, Fv = (x.numpy() for x in self.residual(l + 1, torch.from_numpy(uc), self.mut[l + 1]))
        sc, v = Fc + Fv + self.at * uc + rc, uc
        for _ in range(self.c["gamma"]):
            v = self.fas(l + 1, v, cfl, sc)[0]
        d = np.pad(v - uc, ((0, 0), (1, 1), (1, 1)), mode="edge")
        d[:, 0, 1:-1] = np.where(C.cut, d[:, 1, 1:-1][:, ::-1], d[:, 1, 1:-1])
        d[:, 0, 0], d[:, 0, -1] = d[:, 0, 1], d[:, 0, -2]
        for ax in (1, 2):
            d = np.moveaxis(d, ax, 0)
            e = np.empty((2 * (len(d) - 2),) + d.shape[1:])
            e[0::2], e[1::2] = 0.75 * d[1:-1] + 0.25 * d[:-2], 0.75 * d[1:-1] + 0.25 * d[2:]
            d = np.moveaxis(e, 0, ax)
        return u + d, norm

    def cycles(self, u, first, count):
        norms = []
        for k in range(first, first + count):
            if self.turb:
                self.mut[0] = self.eddy(u)
            cfl = min(self.c["cfl"], RAMP) if k < RAMP_CYCLES else self.c["cfl"]
            u, n = self.fas(0, u, cfl, 0.0)
            norms.append(n)
        return u, np.array(norms)


def exact(case, seed):
    members = _inputs(case, seed)
    m, g, u, v = members[0]
    kind = case["kind"]
    if kind == "batch":
        got = [_Exact(m, g).cycles(u, RAMP_CYCLES, 1) for m, g, u, _ in members]
        return [np.array([n[0] for _, n in got])] + [x for x, _ in got]
    if kind == "pitch":
        dt = 2.0 * math.pi / OMEGA / STEPS
        e = _Exact(m, g, -AMP * math.sin(OMEGA * dt), -AMP * OMEGA * math.cos(OMEGA * dt))
        e.at, e.src = 1.0 / dt, -u / dt
        return list(e.cycles(u, 0, case["count"]))
    e = _Exact(m, g)
    if kind == "residual":
        Fc, Fv = (x.numpy() for x in e.residual(0, torch.from_numpy(u), e.mut[0]))
        return [Fc + Fv, Fc, Fv, math.sqrt(float(np.mean((Fc[0] + Fv[0]) ** 2)))]
    if kind == "precond":
        return [e.sgs(e.lev[0], e.factor(0, u, case["cfl"], e.mut[0])[1], v)]
    if kind == "smooth":
        for _ in range(case["count"]):
            u = e.smooth(0, u, case["cfl"], 0.0)[0]
        return [u]
    if kind == "cycle":
        return list(e.cycles(u, RAMP_CYCLES if case["count"] == 1 else 0, case["count"]))
    mut = [e.eddy(u)] if e.turb else []     # adjoint: J^T v by reverse-mode differentiation of F
    t = torch.from_numpy(u).requires_grad_(True)
    Fc, Fv = e.residual(0, t, mut[0] if e.turb else e.mut[0])
    (jtv,) = torch.autograd.grad(Fc + Fv, t, torch.from_numpy(v))
    return [jtv, None] + mut
