"""What the framework's users have it do, as cases that can be timed and checked.

A pass is a short solve through the public calls: fields in
(lbm_init_fields_pressure), K time steps (lbm_step, or lbm_batch_run of a
plan over several solves), fields and populations out (lbm_moments,
lbm_get_populations, and lbm_diagnostics where a flame is followed).  Every
pass starts from the same initial fields, so it can be repeated.  K is chosen
so that the steps are nearly all of a pass, as they are of a real solve.

Initial states are partly burnt: a progress variable follows each workload's
temperature, every species is present (radicals included), and composition,
velocity and temperature carry seeded noise, so that diffusion, reactions and
all boundary procedures work on values like those of a developed flow.

Outputs are snapshots in the type that holds what a storage resolves: FP64
solves return FP64 arrays; FP32 storage its populations as stored (by
lbm_get_planes over the whole grid), FP32 fields and the velocity, small
against the lattice speed and so resolved to about 1e-4, in FP16; FP16 storage
FP16 fields (the energy in MJ/kg).

`exact` restates the method in plain FP64 torch.
"""
import math

import numpy as np
import torch

from lbm_workloads import fields
from lbm_workloads.mechanism import binary_inert, h2_air_synthetic, with_viscosity_model
from paper_2108_07605_gb300 import lbm

R_U, T0, P0 = 8.314462618, 298.15, 101325.0


# ---- the cases ---------------------------------------------------------------
def listed():
    def case(name, kind, nx, ny, nz, precision, steps, **more):
        return dict(name=name, kind=kind, nx=nx, ny=ny, nz=nz, precision=precision, steps=steps,
                    **more)
    return [
        # the homogeneous reactor at its stated size: the smallest solve, all
        # launches and latency
        case("reactor_16_fp64", "reactor", 16, 16, 16, "fp64", 40, dx_um=1000.0),
        case("reactor_16_fp32", "reactor", 16, 16, 16, "fp32", 40, dx_um=1000.0),
        # the quasi-1D flame at its stated size, followed by its diagnostics
        case("flame_1024_fp64", "flame", 1024, 4, 4, "fp64", 40, diagnostics=True),
        case("flame_1024_fp32", "flame", 1024, 4, 4, "fp32", 60),
        # the 2-D microchannel, in the paper's precision and as its
        # configuration names it: FP32 populations, FP64 chemistry
        case("channel_2000_fp64", "channel", 2000, 40, 1, "fp64", 20),
        case("channel_2000_fp32c64", "channel", 2000, 40, 1, "fp32c64", 40),
        # an odd-sized box without walls, Wilke viscosity, four sub-steps:
        # tails of every tile, between the small and the large grids
        case("box_61x37x29_fp64", "box", 61, 37, 29, "fp64", 16, wilke=True, substeps=4),
        # the 3-D microtube at its stated size in the three storages (FP64 is
        # the headline of bench.py)
        case("tube_600_fp64", "tube", 600, 40, 40, "fp64", 10),
        case("tube_600_fp32", "tube", 600, 40, 40, "fp32", 24),
        case("tube_600_fp16", "tube", 600, 40, 40, "fp16", 24),
        # requests of the serving mix advanced together by one batch plan: a
        # few small ones in FP64, a tick's worth of uneven ones in FP32
        dict(name="batch_small_fp64", kind="batch", precision="fp64", steps=20,
             members="reactor:16 reactor:23 flame:256x4 flame:512x4 reactor:29 flame:1024x4"),
        dict(name="batch_mixed_fp32", kind="batch", precision="fp32", steps=24,
             members="reactor:31 flame:1024x8 reactor:18 flame:512x16 flame:256x32 reactor:25 "
                     "flame:256x8"),
    ]


PRECISIONS = ("fp64", "fp32", "fp32c64", "fp16")
# node-steps of one pass (fluid or not) that a drawn case stays below, by
# lattice and precision (about half of the FP64 tube's time)
MOST_NODE_STEPS = {"fp64": 3e6, "fp32": 1.2e7, "fp32c64": 8e6, "fp16": 1.2e7}


def draw(rng):
    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    kind = rng.choice(("reactor", "flame", "channel", "tube", "box", "batch"))
    # FP16 offsets resolve flows of the order of 1 m/s, not a reactor's rest
    precision = rng.choice(PRECISIONS if kind in ("channel", "tube", "box") else
                           PRECISIONS[:2] if kind == "batch" else PRECISIONS[:3])
    c = dict(kind=kind, precision=precision)
    if kind == "batch":
        members = []
        for _ in range(rng.randint(2, 8)):
            if rng.random() < 0.5:
                members.append("reactor:%d" % size(8, 32))
            else:
                members.append("flame:%dx%d" % (size(64, 1024), size(3, 16)))
        c["members"] = " ".join(members)
        nodes = sum(int(np.prod(s)) for _, s in _members(c))
    else:
        if kind == "reactor":
            n = size(8, 48)
            shape = (n, n, n)
        elif kind == "flame":
            n = size(3, 24)
            shape = (size(64, 1500), n, n)
        elif kind == "channel":
            shape = (size(150, 4000), size(16, 80), 1)
        elif kind == "tube":
            n = size(15, 48)
            shape = (size(24, 500), n, n)
            c["offgrid"] = rng.random() < 0.5
        else:
            flat = rng.random() < 0.25
            shape = (size(5, 120), size(3, 60), 1 if flat else size(3, 60))
            if flat:
                c["lattice"] = "D2Q9"
            c["binary"] = rng.random() < 0.2
            c["wilke"] = not c["binary"] and rng.random() < 0.4
        c["nx"], c["ny"], c["nz"] = shape
        c["substeps"] = rng.choice((1, 2, 2, 4))
        c["diagnostics"] = precision == "fp64" and rng.random() < 0.4
        nodes = int(np.prod(shape))
    c["steps"] = max(2, min(60, int(MOST_NODE_STEPS[precision] / 2 / nodes)))
    return c


def _members(c):
    """[(kind, (nx, ny, nz)), ...] of a batch."""
    out = []
    for m in c["members"].split():
        kind, s = m.split(":")
        v = [int(x) for x in s.split("x")]
        out.append((kind, (v[0], v[0], v[0]) if kind == "reactor" else (v[0], v[1], v[1])))
    return out


# ---- inputs --------------------------------------------------------------------
def _mechanism(c):
    if c.get("binary"):
        return binary_inert(h_formation=(0.0, 1.0e4))
    m = h2_air_synthetic()
    return with_viscosity_model(m, "wilke") if c.get("wilke") else m


def _developed(mech, w, progress, rng):
    """Composition of a workload at the given progress in [0, 1) per node:
    fuel and oxygen consumed in proportion, radicals where the reaction is
    under way, 1 % seeded noise, normalised."""
    i = mech.index
    c = progress
    Y = w["Y"]
    h2 = Y[i("H2")].copy()
    Y[i("H2")] = h2 * (1.0 - 0.95 * c)
    Y[i("O2")] -= 0.95 * c * h2 * 0.5 * mech.molar_mass[i("O2")] / mech.molar_mass[i("H2")]
    Y[i("H2O")] += 0.95 * c * h2 * mech.molar_mass[i("H2O")] / mech.molar_mass[i("H2")]
    zone = 4.0 * c * (1.0 - c)
    for name, most in (("H", 1e-4), ("O", 4e-4), ("OH", 1.5e-3), ("HO2", 6e-5), ("H2O2", 1e-5)):
        Y[i(name)] += most * (zone + 1e-4)
    Y *= 1.0 + 0.01 * rng.uniform(-1.0, 1.0, size=Y.shape)
    Y /= Y.sum(axis=0)


def _workload(mech, c, kind, shape, seed):
    """A workload of lbm_workloads.fields in a developed state."""
    nx, ny, nz = shape
    s = int(seed) & 0x7FFFFFFF
    rng = np.random.Generator(np.random.Philox(key=s + 77))
    if kind == "reactor":
        # 1 mm for the stated reactor, the serving mix's 12.5 um elsewhere
        w = fields.reactor(seed=s, n=nx, dx=c.get("dx_um", 12.5) * 1e-6, mech=mech)
        _developed(mech, w, 0.02 + 0.01 * rng.uniform(-1.0, 1.0, size=w["T"].shape), rng)
        w["u"] += rng.uniform(-0.05, 0.05, size=w["u"].shape)
    elif kind == "flame":
        w = fields.flame_1d(seed=s, nx=nx, ny=ny, nz=nz, x_ign=nx // 4, mech=mech)
        _developed(mech, w, (w["T"] - 300.0) / 1200.0 * 0.98, rng)
    elif kind == "channel":
        w = fields.channel_2d(seed=s, nx=nx, ny=ny, mech=mech)
        _developed(mech, w, 0.3 * ((w["T"] - 300.0) / 1200.0) ** 2, rng)
    elif kind == "tube":
        w = fields.microtube(seed=s, nx=nx, ny=ny, nz=nz, radius=0.475 * ny, mech=mech,
                             offgrid=bool(c.get("offgrid")))
        _developed(mech, w, 0.3 * ((w["T"] - 300.0) / 1200.0) ** 2, rng)
    else:
        binary = bool(c.get("binary"))
        w = fields.perturbed_box(shape, lattice=c.get("lattice", "D3Q27"), seed=s, mech=mech,
                                 amp_u=1.0, T0=300.0 if binary else 1300.0,
                                 dx=2e-7 if binary else 25e-6)
        if binary:
            w["T_max"] = 600.0
        else:
            _developed(mech, w, 0.3 + 0.02 * rng.uniform(-1.0, 1.0, size=w["T"].shape), rng)
    w["substeps"] = int(c.get("substeps", 2))
    return w


def _workloads(c, seed):
    mech = _mechanism(c)
    if c["kind"] == "batch":
        return mech, [_workload(mech, c, k, s, seed * 16 + j)
                      for j, (k, s) in enumerate(_members(c))]
    return mech, [_workload(mech, c, c["kind"], (c["nx"], c["ny"], c["nz"]), seed)]


def _fluid_nodes(kind, shape):
    nx, ny, nz = shape
    if kind != "tube":
        return nx * ny * nz
    solid, _, _ = fields.pipe_wall_geometry(ny, nz, 0.475 * ny)
    return nx * int((~solid).sum())


class _Solve:
    """One handle, its initial fields on the device and its result arrays."""

    def __init__(self, mech, c, w):
        prec = c["precision"]
        bc = {k: w[k] for k in ("faces", "inlet", "outlet", "wall_T", "solid", "solid_kind",
                                "wall_dist", "wall_normal") if k in w}
        self.s = lbm.Solver(mech, lattice=w["lattice"], shape=w["shape"], dx=w["dx"],
                            precision="fp32" if prec == "fp32c64" else prec,
                            chem_fp64=int(prec == "fp32c64"), substeps=w["substeps"],
                            T_max=w["T_max"], **bc)
        self.h, N, M = self.s.h, self.s.N, self.s.M
        self.fields = [torch.from_numpy(np.ascontiguousarray(w[k]).reshape(-1)).cuda()
                       for k in ("P", "u", "T", "Y")]
        f64 = dict(device="cuda", dtype=torch.float64)
        self.out = dict(rho=torch.empty(N, **f64), u=torch.empty(3 * N, **f64),
                        T=torch.empty(N, **f64), Y=torch.empty(M * N, **f64),
                        E=torch.empty(N, **f64))
        self.npop = int(self.s.info.L * self.s.info.Q) * N
        self.storage = "fp32" if prec == "fp32c64" else prec
        self.pops = None
        if self.storage == "fp64":
            self.pops = torch.empty(self.npop, **f64)
        elif self.storage == "fp32":          # the planes hold the T guesses (FP64) behind
            self.pops = torch.empty(self.npop + 2 * N + 2, device="cuda", dtype=torch.float32)
        self.nx = w["shape"][0]

    def init(self):
        lbm.lbm_init_fields_pressure(self.h, *self.fields)

    def result(self):
        lbm.lbm_moments(self.h, **self.out)
        if self.storage == "fp64":
            lbm.lbm_get_populations(self.h, self.pops)
            return dict(self.out, populations=self.pops)
        got = _snapshot(self.out, self.storage)
        if self.storage == "fp32":
            lbm.lbm_get_planes(self.h, 0, self.nx, self.pops)
            got["populations"] = self.pops[:self.npop]
        return got


def _snapshot(out, storage):
    if storage == "fp16":
        return {k: ((v * 1e-6) if k == "E" else v).half() for k, v in out.items()}
    return {k: v.half() if k == "u" else v.float() for k, v in out.items()}


class _State:
    def __init__(self, c, seed):
        mech, ws = _workloads(c, seed)
        self.case = c
        self.solves = [_Solve(mech, c, w) for w in ws]
        self.plan = None
        if c["kind"] == "batch":
            for s in self.solves:       # a plan is made of initialised handles
                s.init()
            self.plan = lbm.lbm_batch_create([s.h for s in self.solves])

    def __del__(self):
        if getattr(self, "plan", None) is not None:
            lbm.lbm_batch_destroy(self.plan)


def prepare(case, seed):
    return _State(case, seed)


def run(state):
    c = state.case
    for s in state.solves:
        s.init()
    if state.plan is not None:
        lbm.lbm_batch_run(state.plan, c["steps"])
        return [s.result() for s in state.solves]
    (s,) = state.solves
    lbm.lbm_step(s.h, c["steps"])
    got = s.result()
    if c.get("diagnostics"):
        got["diagnostics"] = lbm.lbm_diagnostics(s.h)
    return got


# ---- the work a pass cannot do without ------------------------------------------
def work(case):
    """bytes: per fluid node and step every population read once and written
    once, and the initial fields and results once.  flops: per fluid node and
    step, the sums of the moments, the rates of every reaction and sub-step
    (an exponential as 10), the M x M diffusion solve and per population its
    equilibrium, the Stefan-Maxwell sum over the species and the update."""
    s = {"fp64": 8, "fp32": 4, "fp32c64": 4, "fp16": 2}[case["precision"]]
    grids = _members(case) if case["kind"] == "batch" else \
        [(case["kind"], (case["nx"], case["ny"], case["nz"]))]
    M, R = (2, 0) if case.get("binary") else (9, 21)
    D = 2 if case["kind"] == "channel" or case.get("lattice") == "D2Q9" else 3
    Q = 9 if D == 2 else 27
    L = M + 1
    l = int(case.get("substeps", 2))
    out = 8 if s == 8 else s
    nbytes = flops = 0.0
    for kind, shape in grids:
        n = _fluid_nodes(kind, shape)
        N = float(np.prod(shape))
        nbytes += case["steps"] * n * 2.0 * L * Q * s
        nbytes += N * ((5 + M) * 8 + (6 + M) * out + (L * Q * out if s > 2 else 0))
        node = (2 + D) * L * Q + l * R * 44 + 2 * M ** 3 / 3 + 2 * D * M * M + 26 * 2 * (M + D)
        node += Q * (M * 6 + 2 * M * (M - 1) + 5 * (M - 1) + 16)
        flops += case["steps"] * n * node
    return {"bytes": nbytes, "flops": flops}


# ---- the same in 64 bits ---------------------------------------------------------
KIND = {"periodic": 0, "bounce_back": 1, "tms": 2, "inlet": 3, "outlet": 4}
RANK = (0, 3, 3, 2, 1)          # precedence of a boundary kind


class _Exact:
    """The method of arXiv 2108.07605 in plain FP64 torch, step by step:
    streaming, boundary procedures (Sec. 4), moments, temperature, gradients,
    Stefan-Maxwell diffusion velocities, reaction sub-steps, collision."""

    def __init__(self, mech, w):
        self.dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")
        self.mech, self.w = mech, w
        self.D = D = 3 if w["lattice"] == "D3Q27" else 2
        rng = (-1, 0, 1)
        self.c = [(x, y, z) for z in (rng if D == 3 else (0,)) for y in rng for x in rng]
        self.Q = len(self.c)
        self.cv = self.t(np.array(self.c, float)[:, :D])
        self.M = M = mech.n_species
        nx, ny, nz = w["shape"]
        self.ext, self.grid, self.N = (nx, ny, nz), (nz, ny, nx), nx * ny * nz
        self.mm = self.t(mech.molar_mass)
        self.Ra = R_U / self.mm
        self.cref = float(torch.sqrt(self.Ra.max() * w["T_max"] / 0.9))
        self.dx = w["dx"]
        self.dt = self.dx / self.cref
        self.a = self.t(mech.cp_coeffs)
        self.hf, self.s0 = self.t(mech.h_formation), self.t(mech.s_standard)
        self.K = self.t([[0.0 if a == b else 1.0 / (mech.molar_mass[a] * mech.molar_mass[b] *
                                                    mech.D0[a][b]) for b in range(M)]
                         for a in range(M)])
        self.w3 = [math.prod(2 / 3 if v == 0 else 1 / 6 for v in c[:D]) for c in self.c]
        n = torch.arange(self.N, device=self.dev)
        self.xyz = (n % nx, (n // nx) % ny, n // (nx * ny))
        self._boundaries()
        P, T = self.t(w["P"]).reshape(-1), self.t(w["T"]).reshape(-1)
        Y = self.t(w["Y"]).reshape(M, -1)
        u = self.t(w["u"]).reshape(3, -1)[:D] / self.cref
        rho = P / (self.R(Y) * T)
        self.pops = self.equilibria(rho, Y, u, T)
        self.frozen = self.pops[:, :, self.solid].clone()
        self.T = T

    def t(self, v):
        return torch.tensor(np.asarray(v, dtype=np.float64), device=self.dev)

    # thermodynamics
    def R(self, Y):
        return R_U * (Y / self.mm[:, None]).sum(0)

    def H(self, T):
        a = self.a
        poly = (a[:, 0:1] * (T - T0) + a[:, 1:2] / 2 * (T * T - T0 * T0) +
                a[:, 2:3] / 3 * (T ** 3 - T0 ** 3))
        return (self.hf[:, None] + R_U * poly) / self.mm[:, None]

    def U(self, T):
        return self.H(T) - self.Ra[:, None] * T

    def temperature(self, Y, U, T):
        a = self.a
        for _ in range(12):
            cv = (R_U * (a[:, 0:1] + a[:, 1:2] * T + a[:, 2:3] * T * T)) / self.mm[:, None] - \
                self.Ra[:, None]
            dT = ((Y * self.U(T)).sum(0) - U) / (Y * cv).sum(0)
            T = T - dT
            if bool((dT.abs() <= 1e-14 * T.abs()).all()):
                break
        return T

    def rates(self, T, r):
        m, a = self.mech, self.a
        C = r / self.mm[:, None]
        h = self.H(T) * self.mm[:, None]
        s = self.s0[:, None] + R_U * (a[:, 0:1] * torch.log(T / T0) + a[:, 1:2] * (T - T0) +
                                      a[:, 2:3] / 2 * (T * T - T0 * T0))
        g = (h - T * s) / (R_U * T)
        wdot = torch.zeros_like(C)
        for k in range(m.n_reactions):
            A, b, Ea = m.arrhenius[k]
            kf = A * T ** b * torch.exp(-Ea / (R_U * T))
            fwd, rev = kf, torch.zeros_like(kf)
            nu = m.nu_r[k] - m.nu_f[k]
            for j in range(self.M):
                fwd = fwd * C[j] ** int(m.nu_f[k][j])
            if m.reversible[k]:
                Kc = torch.exp(-(self.t(nu)[:, None] * g).sum(0)) * (P0 / (R_U * T)) ** nu.sum()
                rev = kf / Kc
                for j in range(self.M):
                    rev = rev * C[j] ** int(m.nu_r[k][j])
            q = fwd - rev
            if m.third_body[k]:
                q = q * (self.t(m.efficiency[k])[:, None] * C).sum(0)
            for j in range(self.M):
                if nu[j]:
                    wdot[j] += nu[j] * q
        return wdot * self.mm[:, None]

    # equilibria
    @staticmethod
    def psi(c, xi, P):
        return 1.0 - P if c == 0 else 0.5 * (P + c * xi)

    def product(self, u, P):
        return torch.stack([math.prod(self.psi(c[d], u[d], P[d]) for d in range(self.D))
                            for c in self.c])

    def species_eq(self, u, th):
        return self.product(u, th + u * u)

    def energy_eq(self, rho, u, th, U):
        out = []
        for c in self.c:
            A, B = [], []
            for d in range(self.D):
                v = u[d]
                O1, O2 = th * v + v ** 3 / 2, th * th + 2.5 * th * v * v + v ** 4 / 2
                A.append(self.psi(c[d], v, th + v * v))
                B.append(v * v / 2 - O2 if c[d] == 0 else 0.5 * (O2 + c[d] * O1))
            g = U * math.prod(A)
            for d in range(self.D):
                g = g + B[d] * math.prod(A[e] for e in range(self.D) if e != d)
            out.append(rho * g)
        return torch.stack(out)

    def equilibria(self, rho, Y, u, T, us=None):
        c2, M = self.cref ** 2, self.M
        th = self.R(Y) * T / c2
        out = [rho * Y[a] * self.species_eq(u if us is None else us[a], self.Ra[a] * T / c2)
               for a in range(M - 1)]
        out.append(rho * self.species_eq(u, th))
        out.append(self.energy_eq(rho, u, th, (Y * self.U(T)).sum(0) / c2))
        return torch.stack(out)

    # moments of populations [L, Q, n]
    def state(self, p, Tguess):
        M = self.M
        rho, rhoE = p[M - 1].sum(0), p[M].sum(0)
        rs = p[:M - 1].sum(1)
        rs = torch.cat([rs, (rho - rs.sum(0))[None]])
        js = torch.einsum("lqn,qd->ldn", p[:M], self.cv)
        j = js[M - 1].clone()
        js[M - 1] = j - js[:M - 1].sum(0)
        u, Y, E = j / rho, rs / rho, rhoE / rho
        bad = (rs <= 1e-300) | (js.abs() >= rs[:, None]).any(1)
        us = torch.where(bad[:, None], u[None], js / torch.where(bad, torch.ones_like(rs), rs)[:, None])
        T = self.temperature(Y, (E - 0.5 * (u * u).sum(0)) * self.cref ** 2, Tguess)
        return rho, u, Y, us, T, E, rs

    # boundary layout
    def index(self, xyz):
        return xyz[0] + self.ext[0] * (xyz[1] + self.ext[1] * xyz[2])

    def _boundaries(self):
        w, D = self.w, self.D
        self.faces = [KIND[f] for f in w.get("faces", ("periodic",) * 6)]
        solid = w.get("solid")
        self.solid = torch.zeros(self.N, dtype=torch.bool, device=self.dev) if solid is None else \
            torch.as_tensor(np.asarray(solid, bool).reshape(-1), device=self.dev)
        self.walls = any(self.faces) or solid is not None
        rank = torch.tensor(RANK, device=self.dev)
        self.kind = torch.zeros(self.N, dtype=torch.long, device=self.dev)
        self.inc = torch.zeros((self.Q, self.N), dtype=torch.bool, device=self.dev)
        self.src, self.nbr, self.ghost = [], [], []
        for q, c in enumerate(self.c):
            for sign, store in ((-1, self.src), (1, self.nbr)):
                pos, kd = [], torch.zeros_like(self.kind)
                for d in range(3):
                    v = self.xyz[d] + sign * (c[d] if d < D else 0)
                    for mask, f in ((v < 0, 2 * d), (v >= self.ext[d], 2 * d + 1)):
                        fk = self.faces[f]
                        if fk:      # links keep the highest precedence, ghosts the first face
                            take = mask & (RANK[fk] > rank[kd]) if sign < 0 else mask & (kd == 0)
                            kd = torch.where(take, torch.full_like(kd, fk), kd)
                    pos.append(v % self.ext[d])
                at = self.index(pos)
                kd = torch.where((kd == 0) & self.solid[at],
                                 torch.full_like(kd, KIND[w.get("solid_kind", "tms")]), kd)
                store.append(at)
                if sign < 0:
                    self.inc[q] = (kd != 0) & ~self.solid
                    better = rank[kd] > rank[self.kind]
                    self.kind = torch.where(better, kd, self.kind)
                else:
                    self.ghost.append(kd)
        self.kind[self.solid] = 0
        if "inlet" in w:
            u = np.asarray(w["inlet"]["u"], float)
            u = np.broadcast_to(u.reshape(3, 1), (3, self.N)) if u.ndim == 1 else u.reshape(3, -1)
            self.u_in = self.t(u)[:D] / self.cref
            self.T_in = float(w["inlet"]["T"])
            self.Y_in = self.t(w["inlet"]["Y"])
            self.rho_in = float(w["inlet"]["P"] / (self.R(self.Y_in[:, None])[0] * self.T_in))
        if "wall_T" in w:
            self.wall_T = self.t(w["wall_T"]).reshape(-1)

    def reconstruct(self, post, p):
        opp = torch.arange(self.Q - 1, -1, -1, device=self.dev)
        for k in (2, 3, 4):
            i = torch.nonzero(self.kind == k)[:, 0]
            if not len(i):
                continue
            pulled, inc, Tg = p[:, :, i], self.inc[:, i][None], self.T[i]
            if k == 2:
                new = self._wall(pulled, post[:, opp][:, :, i], inc, i, Tg, post)
            elif k == 3:
                new = self._inlet(pulled, inc, i, Tg)
            else:
                new = self._outlet(pulled, inc, i, Tg, post)
            p[:, :, i] = new
        return p

    def _wall(self, p, back, inc, i, Tg, post):
        M = self.M
        pb = torch.where(inc, back, p)
        rho = pb[M - 1].sum(0)
        Y = pb[:M - 1].sum(1) / rho
        Y = torch.cat([Y, (1 - Y.sum(0))[None]])
        u = torch.zeros((self.D, len(i)), dtype=torch.float64, device=self.dev)
        T, us = self.wall_T[i].clone(), None
        if "wall_dist" in self.w:
            nrm = self.t(self.w["wall_normal"]).reshape(3, -1)[:self.D, i]
            dist = self.t(self.w["wall_dist"]).reshape(-1)[i]
            length = self.cv.norm(dim=1)
            dots = (self.cv @ nrm) / torch.where(length > 0, length, torch.ones_like(length))[:, None]
            dots[length == 0] = -math.inf
            best = torch.argmax(dots, 0)
            far = torch.stack(self.nbr)[best, i]
            outside = torch.stack(self.ghost)[best, i] != 0
            h = (self.cv[best] * nrm.T).sum(1)
            _, uf, _, usf, Tf, _, _ = self.state(post[:, :, far], Tg)
            share = torch.where(outside, torch.zeros_like(h), dist / (h + dist))
            u = share * uf
            us = share * usf
            T = torch.where(outside, T, (h * T + dist * Tf) / (h + dist))
        tgt = self.equilibria(rho, Y, u, T, us)
        rl, ul, Yl, usl, Tl, _, _ = self.state(torch.where(inc, tgt, p), Tg)
        loc = self.equilibria(rl, Yl, ul, Tl, usl)
        return torch.where(inc, 2 * tgt - loc, tgt + p - loc)

    def _inlet(self, p, inc, i, Tg):
        one = torch.ones(len(i), dtype=torch.float64, device=self.dev)
        u = self.u_in[:, i]
        fin = self.equilibria(self.rho_in * one, self.Y_in[:, None] * one, u, self.T_in * one)
        rl, ul, Yl, _, Tl, _, _ = self.state(torch.where(inc, fin, p), Tg)
        loc = self.equilibria(rl, Yl, ul, Tl)
        tgt = self.equilibria(rl, Yl, u, self.T_in * one)
        return torch.where(inc, tgt + fin - loc, tgt + p - loc)

    def _outlet(self, p, inc, i, Tg, post):
        """LODI data from the stored state at x and x - n; the cases' outlets
        are the +x face."""
        c2 = self.cref ** 2
        r0, u0, Y0, _, t0, _, _ = self.state(post[:, :, i], Tg)
        r1, u1, Y1, _, t1, _, _ = self.state(post[:, :, i - 1], self.T[i - 1])
        R0 = self.R(Y0)
        p0, p1 = r0 * R0 * t0 / c2, r1 * self.R(Y1) * t1 / c2
        a = self.a
        cv = (Y0 * (R_U * (a[:, 0:1] + a[:, 1:2] * t0 + a[:, 2:3] * t0 * t0) / self.mm[:, None] -
                    self.Ra[:, None])).sum(0)
        cs = torch.sqrt((cv + R0) / cv * R0 * t0 / c2)
        un, un1 = u0[0], u1[0]
        K = 0.25 * (1 - (un / cs) ** 2) * cs / self.ext[0]
        L1 = K * (p0 - float(self.w["outlet"]["P"]) / c2)
        L2 = un * (cs * cs * (r0 - r1) - (p0 - p1))
        L5 = (un + cs) * ((p0 - p1) + r0 * cs * (un - un1))
        ro = r0 - (L2 + 0.5 * (L5 + L1)) / cs ** 2
        po = p0 - 0.5 * (L5 + L1)
        uo = u0 - un * (u0 - u1)
        uo[0] = un - (L5 - L1) / (2 * r0 * cs)
        Yo = Y0 - un * (Y0 - Y1)
        To = po * c2 / (ro * self.R(Yo))
        out = self.equilibria(ro, Yo, uo, To)
        rl, ul, Yl, _, Tl, _, _ = self.state(torch.where(inc, out, p), Tg)
        loc = self.equilibria(rl, Yl, ul, Tl)
        return torch.where(inc, 2 * out - loc, out + p - loc)

    def gradients(self, phi, y):
        """3 sum_i w_i c_i phi_d(x + c_i) of each phi_d along d, and of y along
        every axis, with the ghost values beyond faces and in solids."""
        dphi = torch.zeros_like(phi)
        dy = torch.zeros((self.D,) + y.shape, dtype=torch.float64, device=self.dev)
        if "inlet" in self.w:
            th = float(self.R(self.Y_in[:, None])[0]) * self.T_in / self.cref ** 2
            phi_in = self.rho_in * self.u_in * (1 - 3 * th) - self.rho_in * self.u_in ** 3
        for q, c in enumerate(self.c):
            if not any(c):
                continue
            pv, yv = phi[:, self.nbr[q]], y[:, self.nbr[q]]
            if self.walls:
                g = self.ghost[q]
                pv = torch.where((g == 1) | (g == 2), torch.zeros_like(pv), pv)
                if "inlet" in self.w:
                    pv = torch.where(g == 3, phi_in, pv)
                pv = torch.where(g == 4, phi, pv)
                yv = torch.where(g > 0, y, yv)
            for d in range(self.D):
                if c[d]:
                    dphi[d] += 3 * self.w3[q] * c[d] * pv[d]
                    dy[d] += 3 * self.w3[q] * c[d] * yv
        return dphi, dy

    def step(self):
        M, D, c2, mech = self.M, self.D, self.cref ** 2, self.mech
        post = self.pops
        p = torch.empty_like(post)
        for q in range(self.Q):
            p[:, q] = post[:, q][:, self.src[q]]
        if self.walls:
            p = self.reconstruct(post, p)
        rho, u, Y, us, T, E, rs = self.state(p, self.T)
        # solid nodes hold a state of their own; they are put back at the end
        self.T = T = torch.where(self.solid, self.T, T)
        f, g = p[M - 1], p[M]
        q_g = self.cv.T @ g
        Pten = torch.einsum("qn,qa,qb->abn", f, self.cv, self.cv)
        Ulat = E - 0.5 * (u * u).sum(0)
        th, tha = self.R(Y) * T / c2, self.Ra[:, None] * T / c2
        # relaxation (Sec. 2.3, 3.5)
        s = R_U ** 2 * self.dx / (self.cref * P0) * rho * T * T * (T / T0) ** -mech.D_T_exponent
        ita = s * (self.K @ Y)
        beta = ita / (2 + ita)
        scale = (T / T0) ** mech.mu_T_exponent
        mu = mech.mu0 * scale
        if mech.viscosity_model == "wilke":
            v, ma = self.t(mech.mu0_species), self.mm
            r = (1 + torch.sqrt(v[:, None] / v[None]) * (ma[None] / ma[:, None]) ** 0.25) ** 2 / \
                torch.sqrt(8 * (1 + ma[:, None] / ma[None]))
            X = Y / self.mm[:, None]
            mu = (X * v[:, None] / (r @ X)).sum(0) * scale
        nu = mu / rho / (self.cref * self.dx)
        om = 1 / (nu / th + 0.5)
        om1 = 1 / (nu / mech.prandtl / th + 0.5)
        phi = rho * u * (1 - 3 * th) - rho * u ** 3
        dphi, dy = self.gradients(phi, Y)
        # diffusion velocities (Eq. transform1), elimination without pivoting
        # (the matrix is diagonally dominant)
        A = [[1 + 0.5 * ita[a] if a == b else -0.5 * Y[b] * s * self.K[a, b] for b in range(M)]
             for a in range(M)]
        V = [us[a] - u for a in range(M)]
        for k in range(M):
            for r in range(k + 1, M):
                e = A[r][k] / A[k][k]
                for b in range(k + 1, M):
                    A[r][b] = A[r][b] - e * A[k][b]
                V[r] = V[r] - e * V[k]
        for k in range(M - 1, -1, -1):
            for b in range(k + 1, M):
                V[k] = V[k] - A[k][b] * V[b]
            V[k] = V[k] / A[k][k]
        V = torch.stack(V)
        # reaction sub-steps at frozen energy (Eq. R3)
        r, Ts = rs.clone(), T
        for k in range(self.w["substeps"]):
            if k:
                Ts = self.temperature(r / rho, Ulat * c2, Ts)
            if mech.n_reactions:
                r = r + self.dt / self.w["substeps"] * self.rates(Ts, r)
        drho = r - rs
        # collision
        new = torch.empty_like(p)
        eq = [self.species_eq(u, tha[b]) for b in range(M)]
        d = [rs[b] * (eq[b] - self.species_eq(u + V[b], tha[b])) for b in range(M)]
        for a in range(M - 1):
            F = sum(self.K[a, b] * d[b] for b in range(M) if b != a) * (s * Y[a])
            new[a] = p[a] + 2 * beta[a] * (rs[a] * eq[a] - p[a]) + (beta[a] - 1) * F + drho[a] * eq[a]
        Pex = th + u * u + (2 - om) / (2 * rho * om) * dphi
        new[M - 1] = f + om * (rho * self.product(u, Pex) - f)
        H = self.H(T) / c2
        Pres = rho * th
        W = []
        for a in range(D):
            uP = sum(u[b] * (Pten[b, a] - rho * u[a] * u[b] - (Pres if a == b else 0.0))
                     for b in range(D))
            W.append((om - om1) * (q_g[a] - rho * u[a] * (E + th) - uP - 0.5 * u[a] * dphi[a]) +
                     om1 * rho * (H * Y * V[:, a]).sum(0) +
                     0.5 * (2 - om1) * Pres * (H * dy[a]).sum(0))
        new[M] = g + om * (self.energy_eq(rho, u, th, Ulat) - g)
        for q, c in enumerate(self.c):
            if sum(v * v for v in c) == 1:
                new[M, q] += 0.5 * sum(c[a] * W[a] for a in range(D))
        new[:, :, self.solid] = self.frozen
        self.pops = new

    def result(self, with_pops, with_diag):
        rho, u, Y, _, T, E, rs = self.state(self.pops, self.T)
        v = torch.zeros((3, self.N), dtype=torch.float64, device=self.dev)
        v[:self.D] = u * self.cref
        out = dict(rho=rho, u=v, T=T, Y=Y, E=E * self.cref ** 2)
        out = {k: x.reshape(-1) for k, x in out.items()}
        if with_pops:
            out["populations"] = self.pops.reshape(-1)
        if with_diag:
            q = -(self.H(T) * self.rates(T, rs)).sum(0)
            q = torch.where(self.solid, torch.zeros_like(q), q)
            fluid = ~self.solid
            at = int(torch.nonzero((q == q[fluid].max()) & fluid)[0])
            out["diagnostics"] = dict(hrr_integral=float(q.sum()) * self.dx ** self.D,
                                      hrr_max=float(q[at]), flame_x=at % self.ext[0] * self.dx,
                                      T_max=float(T[fluid].max()),
                                      u_max=float(v[:, fluid].norm(dim=0).max()))
        return out


def exact(case, seed):
    mech, ws = _workloads(case, seed)
    got = []
    for w in ws:
        e = _Exact(mech, w)
        for _ in range(case["steps"]):
            e.step()
        out = e.result(case["precision"] != "fp16", bool(case.get("diagnostics")))
        if case["precision"] == "fp16":
            out["E"] = out["E"] * 1e-6
        got.append(out)
    return got if case["kind"] == "batch" else got[0]
