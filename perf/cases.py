"""Workloads the speed of this library is measured on.

A case is one call pattern of a user's program: advance a simulation by some
coarse steps and fetch its fields (`advance`), evaluate an objective and its
gradients through the autograd function or `Sim.adjoint` (`gradient`), or save
and restore a state (`restart`), on one of two flows:

  vortex    periodic Taylor-Green-like flow, each level refining the central
            half of the one above (Sec. 4.1 of arXiv:1601.06984; the two-level
            boxes of `workloads.config_tgv2d` / `config_tgv3d` are members);
  obstacle  a circle or sphere in a channel with inlet and outlet and nested
            refinement boxes (Secs. 4.2, 4.3; `workloads.config_cylinder` and
            `config_sphere` are members);
  schafer   the paper's own cylinder channel: parabolic inflow, walls, linearly
            interpolated bounce-back on the cylinder.

Results come back in the width of the simulation's storage, as a program that
runs in 32 or 16 bits keeps them.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_1601_06984_gb300 import autograd, lbm
from paper_1601_06984_gb300 import workloads as W

PRECISION = {"fp64": lbm.FP64, "fp32": lbm.FP32DEV, "bf16": lbm.BF16DEV}
MODE = {"linear": lbm.TIME_LINEAR, "two_layer": lbm.TIME_TWO_LAYER, "diffusive": lbm.TIME_DIFFUSIVE}
BYTES = {"fp64": 8, "fp32": 4, "bf16": 2}
U0 = 0.04          # velocity scale, coarsest level
OMEGA_FINEST = 1.6


def listed():
    return [
        # the smallest refined flow of the tests and the smoke run: what counts
        # is the latency of a step, as in a parameter study on tiny meshes
        dict(name="vortex2d_tiny_fp64", task="advance", flow="vortex", stencil=9, nx=32, ny=32, nz=1, levels=2,
             precision="fp64", mode="linear", force=False, steps=20),
        # the four-level cylinder channel with drag read-back: flow studies
        dict(name="cylinder2d_fp32", task="advance", flow="obstacle", stencil=9, cells=5, levels=4,
             precision="fp32", mode="linear", walls=True, steps=50),
        # the paper's cylinder in FP64: parabolic inflow, interpolated walls,
        # two ghost layers instead of interpolation in time (the paper's mode)
        dict(name="schafer2d_fp64", task="advance", flow="schafer", stencil=9, cells=40, levels=2,
             precision="fp64", mode="two_layer", walls=True, steps=50),
        # the two-level 64^3 Taylor-Green vortex, working set about the size of
        # L2: the ordinary 3D run between two field outputs
        dict(name="vortex3d_fp32", task="advance", flow="vortex", stencil=19, nx=64, ny=64, nz=64, levels=2,
             precision="fp32", mode="linear", force=False, steps=200),
        # FP64 reference run with a body force, ragged box
        dict(name="vortex3d_forced_fp64", task="advance", flow="vortex", stencil=19, nx=52, ny=44, nz=36, levels=2,
             precision="fp64", mode="linear", force=True, steps=20),
        # the five-level sphere at half resolution (1.1e7 elements, far beyond
        # L2): the production run
        dict(name="sphere_fp32", task="advance", flow="obstacle", stencil=19, cells=2, levels=5,
             precision="fp32", mode="linear", walls=False, steps=20),
        # the same flow on four levels in the narrowest storage
        dict(name="sphere_bf16", task="advance", flow="obstacle", stencil=19, cells=2, levels=4,
             precision="bf16", mode="linear", walls=False, steps=50),
        # the paper's 3D stencil in the paper's time mode
        dict(name="vortex3d_q27_fp32", task="advance", flow="vortex", stencil=27, nx=96, ny=80, nz=64, levels=2,
             precision="fp32", mode="two_layer", force=False, steps=50),
        # diffusive scaling: four substeps and four ghost layers per interface
        dict(name="vortex3d_diffusive_fp32", task="advance", flow="vortex", stencil=19, nx=48, ny=48, nz=48, levels=2,
             precision="fp32", mode="diffusive", force=False, steps=50),
        # one iteration of a body-force optimisation through torch.autograd
        dict(name="gradient3d_fp32", task="gradient", flow="vortex", stencil=19, nx=64, ny=64, nz=64, levels=2,
             precision="fp32", mode="linear", force=True, steps=40, keep=20),
        # drag gradient of the paper's obstacle flow in FP64 (with respect to
        # the relaxation rate, the inlet velocity and the initial state)
        dict(name="gradient2d_drag_fp64", task="gradient", flow="obstacle", stencil=9, cells=4, levels=3,
             precision="fp64", mode="linear", walls=False, force=False, steps=20, keep=10),
        # start from macroscopic fields, then a checkpoint written and read back
        dict(name="restart3d_fp32", task="restart", flow="vortex", stencil=19, nx=64, ny=64, nz=64, levels=2,
             precision="fp32", mode="linear", force=False, steps=2),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """Another case of the same ranges: mesh sizes (odd extents too), depths,
    storage types, time modes and step counts of the listed flows."""
    task = rng.choice(["advance"] * 5 + ["gradient"] * 2 + ["restart"])
    flow = rng.choice(["vortex", "vortex", "obstacle"] + (["schafer"] if task == "advance" else []))
    c = dict(task=task, flow=flow, stencil=rng.choice([9, 19, 19, 27] if flow == "vortex" else [9, 9, 19]))
    if flow == "schafer":
        c["stencil"] = 9
    three = c["stencil"] > 9
    c["precision"] = rng.choice(["fp64", "fp32", "fp32", "bf16"] if task == "advance" else ["fp64", "fp32"])
    c["mode"] = rng.choice(["linear", "linear", "two_layer"] + (["diffusive"] if task == "advance" else []))
    if flow == "vortex":
        hi = (96 if task == "advance" else 56) if three else 320
        # diffusive scaling wants room for four ghost layers on each side
        lo = 24 if c["mode"] == "diffusive" else 17
        c.update(nx=_log_int(rng, lo, hi), ny=_log_int(rng, lo, hi), nz=_log_int(rng, lo, hi) if three else 1)
        c["levels"] = rng.choice([1, 2, 2, 3]) if min(c["nx"], c["ny"], c["nz"] if three else 999) >= 32 else 2
        c["force"] = task == "gradient" or rng.random() < 0.3
    elif flow == "obstacle":
        if c["mode"] == "diffusive":
            c["mode"] = "linear"  # these nested boxes leave no room for four ghost layers
        c.update(cells=rng.choice([2, 3] if three else [3, 4, 5, 6]), levels=rng.choice([2, 3] if three else [2, 3, 4]),
                 walls=rng.random() < 0.5, force=False)
    else:
        if c["mode"] == "diffusive":
            c["mode"] = "two_layer"
        c.update(cells=rng.choice([20, 40, 60, 80]), levels=2, walls=True, force=False)
    big = three and c["precision"] == "fp64"
    c["steps"] = 2 if task == "restart" else _log_int(rng, 6, 16) if task == "gradient" else _log_int(rng, 10, 20 if big else 60)
    if c["mode"] == "diffusive":
        c["steps"] = max(4, c["steps"] // (1 << c["levels"]))
    if task == "gradient":
        c["keep"] = rng.choice([4, 5, 10])
    return c


# ----------------------------------------------------------------- geometry and inputs
def _boxes(case):
    """(d, extent, boxes [(lo, hi)] in each refined level's cells, bc, ball (centre, radius) or None)."""
    d = 2 if case["stencil"] == 9 else 3
    if case["flow"] == "vortex":
        ext = (case["nx"], case["ny"], case["nz"])[:d]
        boxes, lo, hi = [], (0,) * d, ext
        for _ in range(1, case["levels"]):
            w = [b - a for a, b in zip(lo, hi)]
            lo, hi = (tuple(2 * (a + n // 4) for a, n in zip(lo, w)), tuple(2 * (b - n // 4) for b, n in zip(hi, w)))
            boxes.append((lo, hi))
        return d, ext, boxes, (W.BC_PERIODIC,) * (2 * d), None
    if case["flow"] == "schafer":
        D = case["cells"]
        bc = (W.BC_VELOCITY_IN, W.BC_PRESSURE_OUT, W.BC_WALL, W.BC_WALL)
        return 2, (11 * D, 41 * D // 20), [((D // 2,) * 2, (7 * D // 2,) * 2)], bc, ((2.0 * D,) * 2, 0.5 * D)
    n = case["cells"]
    size = (40, 20) if d == 2 else (32, 16, 16)
    nested = ([((5, 5), (25, 15)), ((7.5, 7.5), (17.5, 12.5)), ((8.5, 8.75), (13.5, 11.25))] if d == 2 else
              [((2, 2, 2), (28, 14, 14)), ((4, 3.5, 3.5), (24, 12.5, 12.5)), ((5, 4.5, 4.5), (20, 11.5, 11.5)),
               ((6, 5.5, 5.5), (16, 10.5, 10.5))])[:case["levels"] - 1]
    # whole cells of the parent level
    boxes = [tuple(tuple(2 * int(round(v * n * (1 << k))) for v in c) for c in b) for k, b in enumerate(nested)]
    D = n << (case["levels"] - 1)
    lateral = W.BC_WALL if case["walls"] else W.BC_PERIODIC
    bc = (W.BC_VELOCITY_IN, W.BC_PRESSURE_OUT) + (lateral,) * (2 * d - 2)
    centre = (10.0 * D, 10.0 * D) if d == 2 else (8.0 * D,) * 3
    return d, tuple(s * n for s in size), boxes, bc, (centre, 0.5 * D)


def _key(case):
    return tuple(sorted((k, v) for k, v in case.items() if k not in ("name", "task", "steps", "keep", "precision")))


@functools.lru_cache(maxsize=4)
def _mesh(key):
    d, ext, boxes, bc, ball = _boxes(dict(key))
    solid = None
    if ball:
        centre, r = np.array(ball[0]), ball[1]

        def solid(L, cen):
            return ((cen - centre) ** 2).sum(axis=1) < r * r

    lmin = int(math.ceil(math.log2(max(ext))))
    return W.nested_boxes(d, lmin, ext, boxes, bc, solid)


def _omega(case):
    return 1.8 if case["mode"] == "diffusive" else W.omega_coarse_from_finest(OMEGA_FINEST, case["levels"])


def _fields(case, mesh, seed):
    """rho, u, S at the elements, in each level's lattice units."""
    rng = np.random.default_rng([W.SEED, seed])
    ns = 3 if mesh.d == 2 else 6
    if case["flow"] == "vortex":
        # divergence-free vortex of random phase and amplitude, extruded in z
        x = mesh.centres()
        kx, ky = 2 * math.pi / mesh.extent[0], 2 * math.pi / mesh.extent[1]
        X, Y = kx * x[:, 0] + rng.uniform(0, 6.28), ky * x[:, 1] + rng.uniform(0, 6.28)
        a = U0 * rng.uniform(0.5, 1.0) / max(kx, ky)
        u = np.zeros((mesh.n, mesh.d))
        u[:, 0], u[:, 1] = -a * ky * np.cos(X) * np.sin(Y), a * kx * np.sin(X) * np.cos(Y)
        if mesh.d == 3:
            u[:, 2] = 0.3 * U0 * np.sin(X + Y)
        S = np.zeros((mesh.n, ns))
        S[:, 0] = a * kx * ky * np.sin(X) * np.sin(Y)
        S[:, 1] = -S[:, 0]
        S *= np.ldexp(1.0, -(mesh.levels.astype(np.int64) - mesh.lmin))[:, None]
        rho = 1.0 - 0.75 * U0 * U0 * (np.cos(2 * X) + np.cos(2 * Y))
    else:
        rho, u, S = W.uniform_fields(mesh, 1.0, (U0, 0.0, 0.0))
        u += 1e-3 * U0 * rng.standard_normal(u.shape)
    if case["mode"] == "diffusive":
        rho, u, S = W.diffusive_units(mesh, rho, u, S)
    return rho, u, S


def _inputs(case, seed):
    mesh = _mesh(_key(case))
    df = None
    if mesh.n < 1_000_000:
        df = W.pdf_perturbation(mesh, case["stencil"], 1e-6, seed=W.SEED + seed)
    force = W.gaussian_force(mesh, 1e-6, seed=W.SEED + seed) if case["force"] else None
    return mesh, _fields(case, mesh, seed) + (df,), force


def _u_in(case):
    return (0.0, 0.0, 0.0) if case["flow"] == "vortex" else (U0, 0.0, 0.0)


# ----------------------------------------------------------------- the measured calls
def prepare(case, seed):
    case = dict(dict(force=False, keep=0), **case)
    mesh, init, force = _inputs(case, seed)
    schafer = case["flow"] == "schafer"
    sim = lbm.Sim(mesh, case["stencil"], _omega(case), precision=PRECISION[case["precision"]], time_mode=MODE[case["mode"]],
                  u_in=_u_in(case), use_force=case["force"], device="cuda" if torch.cuda.is_available() else None,
                  outlet=lbm.OUTLET_ZERO_GRADIENT, bouzidi=schafer,
                  inlet_profile=lbm.INLET_PARABOLIC if schafer else lbm.INLET_UNIFORM)
    if schafer:
        elem, direction = sim.obstacle_links()
        centre, r = _boxes(case)[4]
        sim.set_link_q(W.wall_distance_ball(mesh, elem, direction, centre, r, case["stencil"]))
    state = dict(case=case, sim=sim, init=init,
                 fields=(np.empty(mesh.n), np.empty((mesh.n, mesh.d)), np.empty((mesh.n, 3 if mesh.d == 2 else 6))))
    if case["task"] == "restart":
        return state
    if case["task"] == "gradient" and force is not None:
        dtype = torch.float64 if case["precision"] == "fp64" else torch.float32
        state["force"] = torch.from_numpy(force).to(dtype).requires_grad_()
        state["omega"], state["u_in"] = torch.tensor(_omega(case), dtype=torch.float64), torch.zeros(mesh.d)
        return state
    sim.init(*init)
    if force is not None:
        sim.set_force(force)
    return state


def _width(case, a):
    """A result in the width of the simulation's storage."""
    t = torch.from_numpy(a)
    return t if case["precision"] == "fp64" else t.float() if case["precision"] == "fp32" else t.bfloat16()


def run(state):
    case, sim = state["case"], state["sim"]
    if case["task"] == "restart":
        sim.init(*state["init"])
        sim.step(case["steps"])
        saved = sim.get_state()
        sim.set_state(saved)
        return {"f": _width(case, saved), "totals": _width(case, sim.reduce())}
    if case["task"] == "gradient" and case["force"]:
        state["force"].grad = None
        J = autograd.objective(state["force"], state["omega"], state["u_in"], sim, state["init"], case["steps"], case["keep"])
        J.backward()
        return {"J": J.detach().to(state["force"].dtype), "force": state["force"].grad}
    if case["task"] == "gradient":
        sim.init(*state["init"])
        J, _, dw, du, df0 = sim.adjoint(case["steps"], case["keep"], 1, want_force=False, want_f0=True)
        return {"J": J, "omega": dw, "u_in": du, "f0": df0} if case["precision"] == "fp64" else {"f0": _width(case, df0)}
    sim.step(case["steps"])
    totals = sim.reduce()
    rho, u, S = sim.moments(state["fields"])
    out = {"totals": _width(case, totals), "rho": _width(case, rho), "u": _width(case, u)}
    if case["precision"] != "bf16":  # bfloat16 storage does not resolve the strain rate
        out["S"] = _width(case, S)
    return out


def work(case):
    mesh = _mesh(_key(dict(dict(force=False), **case)))
    q, s = case["stencil"], BYTES[case["precision"]]
    upd = mesh.updates_per_coarse_step(4 if case["mode"] == "diffusive" else 2) * case["steps"]
    ns = mesh.d * (mesh.d + 1) // 2
    if case["task"] == "gradient":
        # forward (read, write), and a reverse that reads the state again and
        # reads and writes the adjoint once
        return {"bytes": 5.0 * upd * q * s, "flops": 3.0 * 12 * q * upd}
    if case["task"] == "restart":
        io = mesh.n * (1 + mesh.d + ns + 2 * q + q) * 8
        return {"bytes": 2.0 * upd * q * s + io, "flops": 12.0 * q * upd}
    return {"bytes": 2.0 * upd * q * s + mesh.n * (1 + mesh.d + ns) * 8, "flops": 12.0 * q * upd}


# ----------------------------------------------------------------- the same flow in 64 bits on dense arrays
class _Dense:
    """The multilevel method on one dense torch array per level (the refined
    box and a margin of ghost cells), in float64: Secs. 2.1-2.3."""

    def __init__(self, case):
        self.case = case
        self.dev = "cuda" if torch.cuda.is_available() else "cpu"
        self.d, self.ext, boxes, self.bc, self.ball = _boxes(case)
        d, q = self.d, case["stencil"]
        c = (W._C9 if q == 9 else W._C27[:q])[:, :d]
        self.c = [tuple(int(v) for v in r) for r in c]
        n2 = (c ** 2).sum(1)
        table = {9: {0: 4 / 9, 1: 1 / 9, 2: 1 / 36}, 19: {0: 1 / 3, 1: 1 / 18, 2: 1 / 36},
                 27: {0: 8 / 27, 1: 2 / 27, 2: 1 / 54, 3: 1 / 216}}[q]
        self.opp = [0] + [i + 1 if i % 2 else i - 1 for i in range(1, q)]
        self.diffusive = case["mode"] == "diffusive"
        self.m = 4 if self.diffusive else 2
        self.pad = 4 if self.diffusive else 2
        self.pairs = [(a, a) for a in range(d)] + ([(0, 1)] if d == 2 else [(0, 1), (1, 2), (0, 2)])
        self.ct = torch.tensor(c, dtype=torch.float64, device=self.dev)
        self.w = torch.tensor([table[int(n)] for n in n2], dtype=torch.float64, device=self.dev)
        self.lo = [(0,) * d] + [b[0] for b in boxes]
        self.hi = [self.ext] + [b[1] for b in boxes]
        self.nlev = len(self.lo)
        self.org = [tuple(v - (self.pad if k else 0) for v in self.lo[k]) for k in range(self.nlev)]
        self.shape = [tuple(b - a + (2 * self.pad if k else 0) for a, b in zip(self.lo[k], self.hi[k]))
                      for k in range(self.nlev)]
        self.u_in = _u_in(case)[:d]
        self.set_omega(torch.tensor(_omega(case), dtype=torch.float64, device=self.dev))
        self.margin, self.solid, self.q = [], [], []
        for k in range(self.nlev):
            inside = torch.zeros(self.shape[k], dtype=torch.bool, device=self.dev)
            p = self.pad if k else 0
            inside[tuple(slice(p, n - p) for n in self.shape[k])] = True
            self.margin.append(~inside)
            x = [((torch.arange(n, dtype=torch.float64, device=self.dev) + o + 0.5) * (1 << (self.nlev - 1 - k)))
                 .reshape([-1 if a == b else 1 for b in range(d)]) for a, (n, o) in enumerate(zip(self.shape[k], self.org[k]))]
            if self.ball and k == self.nlev - 1:
                r2 = sum((x[a] - self.ball[0][a]) ** 2 for a in range(d))
                self.solid.append(r2 < self.ball[1] ** 2)
                # wall distance along each link
                qs = []
                for ci in self.c:
                    b = sum(-(x[a] - self.ball[0][a]) * ci[a] for a in range(d)) + 0 * r2
                    aa = max(1, sum(v * v for v in ci))
                    qs.append(((-b - torch.sqrt(torch.clamp(b * b - aa * (r2 - self.ball[1] ** 2), min=0.0))) / aa).clamp(1e-6, 1.0))
                self.q = qs
            else:
                self.solid.append(None)

    def set_omega(self, omega):
        self.om = [omega]
        for _ in range(1, self.nlev):
            self.om.append(self.om[-1] if self.diffusive else 1.0 / (0.5 + 2.0 * (1.0 / self.om[-1] - 0.5)))

    # -- pieces
    def col(self, v):
        return v.reshape((-1,) + (1,) * self.d)

    def dot_c(self, u):
        return torch.tensordot(self.ct, u, dims=1)

    def feq(self, rho, u):
        cu = self.dot_c(u)
        return self.col(self.w) * rho * (1 + 3 * cu + 4.5 * cu * cu - 1.5 * (u * u).sum(0))

    def guo(self, om, u, F):
        cu, cF = self.dot_c(u), self.dot_c(F)
        return (1 - 0.5 * om) * self.col(self.w) * (3 * (cF - (u * F).sum(0)) + 9 * cu * cF)

    def stored(self, f, om, F):
        """rho, u, S, f^neq of a stored post-collision state."""
        rho = f.sum(0)
        j = torch.tensordot(self.ct.t(), f, dims=1)
        u = (j if F is None else j - 0.5 * F) / rho
        fn = f - self.feq(rho, u)
        if F is not None:
            fn = fn - self.guo(om, u, F)
        fn = fn / (1 - om)
        S = torch.stack([torch.tensordot(self.ct[:, a] * self.ct[:, b], fn, dims=1) for a, b in self.pairs])
        return rho, u, S * (-1.5 * om / rho), fn

    def stream_collide(self, f, k, F):
        d, s = self.d, self.solid[k]
        g = []
        for i, ci in enumerate(self.c):
            gi = torch.roll(f[i], ci, tuple(range(d))) if i else f[0]
            if i and s is not None:
                wall = torch.roll(s, ci, tuple(range(d)))
                back = f[self.opp[i]]
                if self.case["flow"] == "schafer":
                    away = torch.roll(back, tuple(-v for v in ci), tuple(range(d)))
                    q = self.q[i]
                    back = torch.where(q < 0.5, 2 * q * back + (1 - 2 * q) * away, back / (2 * q) + (2 * q - 1) / (2 * q) * f[i])
                gi = torch.where(wall, back, gi)
            g.append(gi)
        if k == 0 and self.ball:
            g = self.channel(f, g)
        f0, f = f, torch.stack(g)
        rho = f.sum(0)
        j = torch.tensordot(self.ct.t(), f, dims=1)
        u = (j if F is None else j + 0.5 * F) / rho
        out = f + self.om[k] * (self.feq(rho, u) - f)
        if F is not None:
            out = out + self.guo(self.om[k], u, F)
        return out if s is None else torch.where(s, f0, out)

    def channel(self, f, g):
        """Inlet at x-, outlet at x+ (zero gradient), walls or periodic faces elsewhere, on the coarsest level."""
        n = self.shape[0]
        at = lambda a, i: torch.arange(n[a], device=self.dev).reshape([-1 if a == b else 1 for b in range(self.d)]) == i
        rho, u, _, fn = self.stored(f, self.om[0], None)
        eq0 = self.feq(torch.ones_like(rho), u)
        for i, ci in enumerate(self.c[1:], 1):
            if ci[0] > 0:
                prof = 1.0
                if self.case["flow"] == "schafer":
                    t = (torch.arange(n[1], dtype=torch.float64, device=self.dev) + 0.5 - 0.5 * ci[1]) / n[1]
                    prof = (6 * t * (1 - t)).reshape(1, -1)
                term = 6 * self.w[i] * sum(v * x for v, x in zip(ci, self.u_in)) * prof
                g[i] = torch.where(at(0, 0), f[self.opp[i]] + term, g[i])
            elif ci[0] < 0:
                if sum(v * v for v in ci) == 1:
                    val = eq0[i] + fn[self.opp[i]]
                else:
                    val = torch.roll(f[i], ci[1:], tuple(range(1, self.d)))  # f_i(x - c_i - n)
                g[i] = torch.where(at(0, n[0] - 1), val, g[i])
            if self.bc[2] == W.BC_WALL:
                for a in range(1, self.d):
                    if ci[a]:
                        g[i] = torch.where(at(a, 0 if ci[a] > 0 else n[a] - 1), f[self.opp[i]], g[i])
        return g

    def odd_scaled(self, fn, r):
        return fn if not self.diffusive else 0.5 * (fn + fn[self.opp]) + 0.5 * r * (fn - fn[self.opp])

    def restrict(self, fc, ff, k, F):
        """Level k's cells under level k + 1 from their children."""
        p, d, m = self.pad, self.d, self.m
        inner = (slice(None),) + tuple(slice(p, n - p) for n in self.shape[k + 1])
        rho, u, S, fn = self.stored(ff[inner], self.om[k + 1], None if F is None else F[k + 1][inner])
        fn = self.odd_scaled(fn, 2.0)

        def kids(x, axis=None):
            sh = [x.shape[0]]
            for n in x.shape[1:]:
                sh += [n // 2, 2]
            x = x.reshape(sh)
            if axis is not None:
                sgn = torch.tensor([-1.0, 1.0], dtype=torch.float64, device=self.dev)
                x = x * sgn.reshape([2 if b == 2 + 2 * axis else 1 for b in range(x.dim())])
            return x.sum(dim=[2 + 2 * a for a in range(d)])

        n = 1 << d
        dS = [kids(S, a) for a in range(d)]
        si = lambda a, b: self.pairs.index((a, b) if (a, b) in self.pairs else (b, a))
        us = m / 2.0
        um = kids(u) / n * us
        lap = torch.stack([sum(2 * dS[b][si(a, b)] - dS[a][b] for b in range(d)) for a in range(d)])
        um = um - lap * (m * (0.5 if d == 3 else 1.0)) / 32.0
        rm = 1 + us * us * (kids(rho[None])[0] / n - 1)
        wc, wf = self.om[k], self.om[k + 1]
        g = self.feq(rm, um) + (1 - wc) * m * wf / wc * kids(fn) / n
        out = fc.clone()
        out[(slice(None),) + tuple(slice(a // 2 - o, b // 2 - o) for a, b, o in
                                   zip(self.lo[k + 1], self.hi[k + 1], self.org[k]))] = g
        return out

    def records(self, f, k, F):
        rho, u, S, fn = self.stored(f, self.om[k], None if F is None else F[k])
        return torch.cat([rho[None], u, S, fn])

    def prolong(self, ff, rec, k):
        """Level k's margin from level k - 1's source records (compact quadratic interpolation)."""
        d, m = self.d, self.m
        par = [(o // 2, (o + n) // 2) for o, n in zip(self.org[k], self.shape[k])]
        offs = [(0, 0, 0), (1, 1, 0), (1, 0, 1), (0, 1, 1)] if d == 3 else [(0, 0), (1, 0), (0, 1), (1, 1)]
        lw = [0.625, 0.125, 0.125, 0.125] if d == 3 else [0.5625, 0.1875, 0.1875, 0.0625]
        wc, wf = self.om[k - 1], self.om[k]
        out = ff.clone()
        for octant in range(1 << d):
            sg = [1 if (octant >> a) & 1 else -1 for a in range(d)]
            src = [rec[(slice(None),) + tuple(slice(a + s * o - g, b + s * o - g) for (a, b), s, o, g in
                                              zip(par, sg, off, self.org[k - 1]))] for off in offs]
            lin = sum(w * s for w, s in zip(lw, src))
            # velocities and strain rates in the octant's frame
            ul = [[sg[a] * s[1 + a] for a in range(d)] for s in src]
            Sl = [[sg[a] * sg[b] * s[1 + d + t] for t, (a, b) in enumerate(self.pairs)] for s in src]
            dif = lambda t, c: 0.5 * sum(v * s[t] for v, s in zip(c, Sl))
            if d == 3:
                X, Y, Z = (lambda t: dif(t, (-1, 1, 1, -1))), (lambda t: dif(t, (-1, 1, -1, 1))), (lambda t: dif(t, (-1, -1, 1, 1)))
                xx, yy, zz, xy, yz, xz = range(6)
                mix = Z(xy) + X(yz) + Y(xz)
                same = [0.5 * X(xx) + Y(xy) - 0.5 * X(yy) + Z(xz) - 0.5 * X(zz),
                        X(xy) - 0.5 * Y(xx) + 0.5 * Y(yy) + Z(yz) - 0.5 * Y(zz),
                        X(xz) - 0.5 * Z(xx) + Y(yz) - 0.5 * Z(yy) + 0.5 * Z(zz)]
                cross = [Y(xx) + Z(xx) + mix - 2 * X(yz), X(yy) + Z(yy) + mix - 2 * Y(xz), X(zz) + Y(zz) + mix - 2 * Z(xy)]
                loc = [0.625 * ul[0][a] + 0.125 * (ul[1][a] + ul[2][a] + ul[3][a]) - 0.1875 * same[a] - 0.0625 * cross[a]
                       for a in range(3)]
            else:
                X, Y = (lambda t: dif(t, (-1, 1, -1, 1))), (lambda t: dif(t, (-1, -1, 1, 1)))
                same = [0.5 * X(0) + Y(2) - 0.5 * X(1), X(2) - 0.5 * Y(0) + 0.5 * Y(1)]
                cross = [Y(0), X(1)]
                loc = [0.5 * ul[0][a] + 0.25 * (ul[1][a] + ul[2][a]) - 0.1875 * same[a] + 0.0625 * cross[a] for a in range(2)]
            us = 2.0 / m
            u = torch.stack([s * v * us for s, v in zip(sg, loc)])
            rho = 1 + us * us * (lin[0] - 1)
            fn = self.odd_scaled(lin[1 + d + len(self.pairs):], 0.5)
            g = self.feq(rho, u) + (1 - wf) * wc / (m * wf) * fn
            at = (slice(None),) + tuple(slice((octant >> a) & 1, None, 2) for a in range(d))
            out[at] = torch.where(self.margin[k][at[1:]], g, out[at])
        return out

    def advance(self, f, k, F):
        finer = k + 1 < self.nlev
        if finer:
            f[k] = self.restrict(f[k], f[k + 1], k, F)
            rec = self.records(f[k], k, F)
            f[k + 1] = self.prolong(f[k + 1], rec, k + 1)
        f[k] = self.stream_collide(f[k], k, None if F is None else F[k])
        if finer:
            self.advance(f, k + 1, F)
            if self.case["mode"] == "linear":
                f[k + 1] = self.prolong(f[k + 1], 0.5 * (rec + self.records(f[k], k, F)), k + 1)
            for _ in range(1, self.m):
                self.advance(f, k + 1, F)

    # -- between caller order and the arrays
    def index(self, mesh):
        got = []
        for k in range(self.nlev):
            sel = np.flatnonzero(mesh.levels == mesh.lmin + k)
            xyz = mesh.coords[sel] - np.array(self.org[k])
            flat = np.ravel_multi_index(tuple(xyz.T), self.shape[k])
            got.append((torch.from_numpy(sel).to(self.dev), torch.from_numpy(flat).to(self.dev)))
        return got

    def scatter(self, x, k, fill):
        """[n, c] caller-order values on level k's array [c, ...]; `fill` elsewhere."""
        sel, flat = self.where[k]
        out = fill.reshape(-1, 1).expand(-1, math.prod(self.shape[k])).clone()
        return out.index_copy(1, flat, x[sel].t()).reshape((-1,) + self.shape[k])

    def start(self, mesh, rho, u, S, df):
        self.where = self.index(mesh)
        t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(self.dev)
        rho, u, S, df = t(rho), t(u), t(S), None if df is None else t(df)
        f = []
        zero = torch.zeros(1, dtype=torch.float64, device=self.dev)
        for k in range(self.nlev):
            r = self.scatter(rho[:, None], k, zero + 1)[0]
            v, s = self.scatter(u, k, zero.expand(self.d)), self.scatter(S, k, zero.expand(len(self.pairs)))
            qs = sum((1 if a == b else 2) * self.col(self.ct[:, a] * self.ct[:, b]) * s[t] for t, (a, b) in enumerate(self.pairs))
            fk = self.feq(r, v) - (1 - self.om[k]) * 3 * self.col(self.w) * r / self.om[k] * (qs - s[:self.d].sum(0) / 3)
            f.append(fk if df is None else fk + self.scatter(df, k, zero.expand(len(self.c))))
        return f

    def gather(self, parts, n):
        """Per-level arrays [c, ...] in caller order, [n, c]."""
        out = torch.zeros((n, parts[0].shape[0]), dtype=torch.float64, device=self.dev)
        for (sel, flat), p in zip(self.where, parts):
            out[sel] = p.reshape(p.shape[0], -1)[:, flat].t()
        return out

    def reduce(self, f, F):
        d, tot = self.d, 0
        for k in range(self.nlev):
            sel, flat = self.where[k]
            pick = lambda x: x.reshape(x.shape[0], -1)[:, flat]
            g = pick(f[k])
            rho = g.sum(0)
            j = self.ct.t() @ g
            if F is not None:
                j = j - 0.5 * pick(F[k])
            us = 2.0 ** k if self.diffusive else 1.0
            vol = 2.0 ** (-d * k)
            obs = torch.zeros(3, dtype=torch.float64, device=self.dev)
            if self.solid[k] is not None:
                fluid = torch.zeros(math.prod(self.shape[k]), dtype=torch.bool, device=self.dev)
                fluid[flat] = True
                fluid = fluid.reshape(self.shape[k])
                for i, ci in enumerate(self.c[1:], 1):
                    link = torch.roll(self.solid[k], ci, tuple(range(d))) & fluid
                    own = f[k][self.opp[i]]
                    back = own
                    if self.case["flow"] == "schafer":
                        q, away = self.q[i], torch.roll(own, tuple(-v for v in ci), tuple(range(d)))
                        back = torch.where(q < 0.5, 2 * q * own + (1 - 2 * q) * away, own / (2 * q) + (2 * q - 1) / (2 * q) * f[k][i])
                    amount = torch.where(link, own + back, torch.zeros_like(own)).sum()
                    obs = obs + torch.stack([-amount * ci[a] if a < d else 0 * amount for a in range(3)])
            pad = torch.zeros(3 - d, dtype=torch.float64, device=self.dev)
            tot = tot + torch.cat([(vol * (1 + us * us * (rho - 1)).sum())[None], vol * us * j.sum(1), pad, obs,
                                   (vol * us * us * 0.5 * ((j * j).sum(0) / rho).sum())[None]])
        return tot


def exact(case, seed):
    case = dict(dict(force=False, keep=0), **case)
    mesh, (rho, u, S, df), force = _inputs(case, seed)
    if work(case)["bytes"] > (5e11 if case["task"] == "advance" else 1.2e11):
        return None
    s = _Dense(case)
    f = s.start(mesh, rho, u, S, df)
    to_host = lambda x: x.detach().cpu()
    forces = lambda t: None if t is None else [s.scatter(t, k, torch.zeros(s.d, dtype=torch.float64, device=s.dev)) for k in range(s.nlev)]
    if case["task"] != "gradient":
        F = forces(None if force is None else torch.from_numpy(force).to(s.dev))
        with torch.no_grad():
            for _ in range(case["steps"]):
                s.advance(f, 0, F)
            totals = to_host(s.reduce(f, F))
            if case["task"] == "restart":
                return {"f": to_host(s.gather(f, mesh.n)), "totals": totals}
            got = [s.stored(f[k], s.om[k], None if F is None else F[k]) for k in range(s.nlev)]
            out = {"totals": totals, "rho": to_host(s.gather([g[0][None] for g in got], mesh.n))[:, 0],
                   "u": to_host(s.gather([g[1] for g in got], mesh.n))}
            if case["precision"] != "bf16":
                out["S"] = to_host(s.gather([g[2] for g in got], mesh.n))
            return out
    from torch.utils.checkpoint import checkpoint

    def step(*f):
        f = list(f)
        s.advance(f, 0, F)
        return tuple(f)

    omega = torch.tensor(_omega(case), dtype=torch.float64, device=s.dev, requires_grad=True)
    u_in = torch.tensor(_u_in(case)[:s.d], dtype=torch.float64, device=s.dev, requires_grad=True)
    f0 = s.gather([x.detach() for x in f], mesh.n).requires_grad_()
    s.set_omega(omega)
    s.u_in = u_in
    if force is not None:
        force = force if case["precision"] == "fp64" else force.astype(np.float32).astype(np.float64)
        force = torch.from_numpy(force).to(s.dev).requires_grad_()
    F = forces(force)
    f = tuple(s.scatter(f0, k, s.w) for k in range(s.nlev))
    for _ in range(case["steps"]):
        f = checkpoint(step, *f, use_reentrant=False)
    tot = s.reduce(list(f), F)
    J = tot[7] if case["force"] else tot[4]
    J.backward()
    if case["force"]:
        return {"J": to_host(J), "force": to_host(force.grad)}
    if case["precision"] != "fp64":
        return {"f0": to_host(f0.grad)}
    du = None if u_in.grad is None else torch.cat([to_host(u_in.grad), torch.zeros(3 - s.d, dtype=torch.float64)])
    return {"J": float(J), "omega": float(omega.grad), "u_in": du, "f0": to_host(f0.grad)}
