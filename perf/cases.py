"""The work this solver is used for, as cases that a timing program can run.

A pass is what a program that melts a phase-change material does again and
again: advance a run (or a batch of runs) by some hundred time steps through
``Solver.step`` or ``Batch.step``, then take the fields of the new time level
(and, where the run is being monitored, its FP64 diagnostics).  Runs start from
a developed melting state: a hot liquid region with a curved front, a
convection roll at the Darcy velocity, and the foam a little off the melt's
temperature.  The seed draws the front, the roll, and the groups that the batched
workload draws too (porosity, Da, Ra, Ste), about the paper's own.

A 16-bit run's snapshot is kept in the type the run stores its populations in.
"""
import math

import numpy as np
import torch

from paper_1701_00702_gb300 import inputs, lbm

PRECISION = {"f64": 0, "f32": 1, "f16": 2, "bf16": 3}
SNAPSHOT = {"f16": torch.float16, "bf16": torch.bfloat16}
# the fields a batch's owner reads from every run (the benchmark's end-to-end list)
BATCH_FIELDS = ("T_f", "T_s", "f_l", "u_x", "u_y")

# D2Q9 directions (the first five are those of D2Q5) and flow weights
EX = (0, 1, 0, -1, 0, 1, -1, -1, 1)
EY = (0, 0, 1, 0, -1, 1, 1, -1, -1)
W9 = (4 / 9, 1 / 9, 1 / 9, 1 / 9, 1 / 9, 1 / 36, 1 / 36, 1 / 36, 1 / 36)


def _run(name, nx, ny, precision, steps, lattice=5, flow=True, eq9=False, diag=False):
    return dict(name=name, kind="run", nx=nx, ny=ny, precision=precision, steps=steps, lattice=lattice, flow=flow,
                eq9=eq9, diag=diag)


def listed():
    return [
        # the one-dimensional conduction melting of Sec. IV A in its own size and type: the smallest grid
        _run("conduction_200x4_f64", 200, 4, "f64", 500, flow=False),
        # a small cavity watched closely: ten steps, then diagnostics and fields (launches and latency)
        _run("watch_64_f32", 64, 64, "f32", 10, diag=True),
        # the grid of Sec. IV B (and of lbm_params_default)
        _run("cavity_150_f32", 150, 150, "f32", 250),
        # the headline run of the benchmark
        _run("cavity_256_f32", 256, 256, "f32", 200),
        # the same run in the type that reference solutions are made in
        _run("cavity_256_f64", 256, 256, "f64", 50),
        # the D2Q9 thermal lattices of Sec. III B, on an oblong grid
        _run("cavity_300x200_q9_f32", 300, 200, "f32", 150, lattice=9),
        # a middle-sized run in FP16 storage (state within L2)
        _run("cavity_512_f16", 512, 512, "f16", 200),
        # ragged sides, BF16 storage, phase-dependent conductivity and heat capacity (Eq. 9)
        _run("eq9_777x501_bf16", 777, 501, "bf16", 100, eq9=True),
        # a run beyond L2 that is monitored: a few steps, then diagnostics and fields
        _run("watch_1024_f32", 1024, 1024, "f32", 16, diag=True),
        # the large runs, whose state streams through HBM
        _run("cavity_2048_f32", 2048, 2048, "f32", 50),
        _run("cavity_2048_f16", 2048, 2048, "f16", 50),
        # unequal cavities advanced together as the server does (grouped launches, FP16 storage)
        dict(name="batch_12_f16", kind="batch", count=12, n_lo=64, n_hi=512, sides=1701, precision="f16", map=4,
             steps=256),
    ]


def draw(rng):
    def log(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    if rng.random() < 0.15:
        precision = rng.choice(["f16", "bf16", "f32"])
        return dict(kind="batch", count=rng.randint(4, 12), n_lo=64, n_hi=rng.randint(128, 512),
                    sides=rng.randint(0, 9999), precision=precision, map=5 if precision == "f32" else 4,
                    steps=rng.randint(48, 256))
    c = _run("", 0, 0, rng.choice(["f32", "f32", "f32", "f16", "f16", "bf16", "f64"]), 0,
             lattice=9 if rng.random() < 0.2 else 5, eq9=rng.random() < 0.15, diag=rng.random() < 0.25)
    del c["name"]
    if rng.random() < 0.12:   # conduction only: a strip, periodic across
        c.update(flow=False, eq9=False, nx=log(100, 1000), ny=rng.randint(3, 64))
    else:
        top = 320 if c["precision"] == "f64" else 1100 if c["lattice"] == 9 else 2048
        c["nx"] = log(64, top)
        c["ny"] = max(48, min(2048, int(round(c["nx"] * rng.uniform(0.5, 1.0)))))
    # as many steps as keep a pass within the largest listed one's
    room = (2 << 20 if c["precision"] == "f64" else 80 << 20) // (c["nx"] * c["ny"])
    c["steps"] = rng.randint(8, max(12, min(250, room)))
    return c


def _sides(case):
    """Sides of a batch's cavities, uniform in [n_lo, n_hi]; the case's own, whatever the seed of the inputs."""
    rng = np.random.default_rng(case["sides"])
    return [int(n) for n in rng.integers(case["n_lo"], case["n_hi"] + 1, case["count"])]


def _groups(rng):
    """Non-dimensional groups about those of Sec. IV B (Da = 1e-4, Ra = 1e6, Ste = 1)."""
    return dict(porosity=float(rng.uniform(0.85, 0.98)), Da=float(1e-4 * 10 ** rng.uniform(0, 1)),
                Ra=float(5e5 * 4 ** rng.uniform(0, 1)), Ste=float(rng.uniform(0.5, 2.0)))


def _parameters(case, seed):
    """The parameter sets of a case's runs (one for a single run)."""
    prec = PRECISION[case["precision"]]
    rng = np.random.default_rng([seed, 1])
    if case["kind"] == "batch":
        return [inputs.cavity(n, precision=prec, **_groups(rng)) for n in _sides(case)]
    if not case["flow"]:
        return [inputs.conduction_1d(case["nx"], case["ny"], precision=prec, thermal_q=case["lattice"],
                                     porosity=float(rng.uniform(0.85, 0.98)), Ste=float(rng.uniform(0.5, 2.0)))]
    over = _groups(rng)
    if case["eq9"]:
        over.update(ks_over_kl=float(rng.uniform(0.5, 1.5)), cps_over_cpl=float(rng.uniform(0.8, 1.2)))
    return [inputs.cavity(case["nx"], ny=case["ny"], precision=prec, thermal_q=case["lattice"], **over)]


# ---------------------------------------------------------------------------
# A developed melting state, in float64 on the GPU
# ---------------------------------------------------------------------------

class _Constants:
    """Lattice-unit constants of a parameter set (Eq. 54 and Sec. III C)."""

    def __init__(self, p):
        self.p = p
        L, dT, phi = p["L_char"], p["T_hot"] - p["T_cold"], p["porosity"]
        self.phi, self.Q = phi, p["thermal_q"]
        self.nu = p["Pr"] * p["k_f"]
        self.gbeta = p["Ra"] * self.nu * p["k_f"] / (dT * L ** 3)
        self.K = p["Da"] * L * L
        self.k_m, self.rho_m = p["cond_ratio"] * p["k_f"], p["sigma_hat"]
        self.h_v = p["Nu_i"] * p["k_f"] / (p["dp_over_L"] * L) ** 2
        self.c_ps, self.k_s = p["cps_over_cpl"], p["ks_over_kl"] * p["k_f"]
        self.H_fs = self.c_ps * p["T_solidus"]
        self.H_fl = p["T_liquidus"] + dT / p["Ste"]
        self.cs2 = 1 / 3 if self.Q == 9 else 0.5 * p["varpi"]
        # equilibrium weights of the moving thermal populations, and their sum
        self.w = W9 if self.Q == 9 else (0.0,) + (0.25 * p["varpi"],) * 4
        self.wsum = 5 / 9 if self.Q == 9 else p["varpi"]
        self.eta = 1 / (0.5 + self.k_m / (self.rho_m * p["cmref_over_cpm"] * self.cs2))

    def enthalpy(self, T):
        p = self.p
        if T <= p["T_solidus"]:
            return self.c_ps * T
        if T >= p["T_liquidus"]:
            return self.H_fl + T - p["T_liquidus"]
        return self.H_fs + (T - p["T_solidus"]) / (p["T_liquidus"] - p["T_solidus"]) * (self.H_fl - self.H_fs)

    def state_of(self, H):
        p = self.p
        fl = ((H - self.H_fs) / (self.H_fl - self.H_fs)).clamp(0, 1)
        T = (H / self.c_ps).clamp(max=p["T_solidus"]) + fl * (p["T_liquidus"] - p["T_solidus"])
        return T + (H - self.H_fl).clamp(min=0), fl

    def f_eq(self, rho, ux, uy):
        uu = ux * ux + uy * uy
        out = []
        for i in range(9):
            eu = EX[i] * ux + EY[i] * uy
            out.append(W9[i] * rho * (1 + 3 * eu + (4.5 * eu * eu - 1.5 * uu) / self.phi))
        return torch.stack(out)

    def g_eq(self, H, T, ux, uy):
        c = self.p["cfref_over_cpl"]
        out = [H - self.wsum * c * T]
        for i in range(1, self.Q):
            out.append(self.w[i] * T * (c + (EX[i] * ux + EY[i] * uy) / (self.phi * self.cs2)))
        return torch.stack(out)

    def h_eq(self, T):
        c = self.p["cmref_over_cpm"]
        return torch.stack([T - self.wsum * c * T] + [self.w[i] * c * T for i in range(1, self.Q)])


def _melting(p, seed):
    """Populations f - w, g, h and the history T_m - T_f of a developed state, in the run's own real type."""
    c = _Constants(p)
    rng = np.random.default_rng([seed, 2])
    nx, ny = p["nx"], p["ny"]
    y, x = torch.meshgrid(torch.arange(ny, dtype=torch.float64, device="cuda"),
                          torch.arange(nx, dtype=torch.float64, device="cuda"), indexing="ij")
    s = (2 * math.pi if p["periodic_y"] else math.pi) * (y + 0.5) / ny
    front = (nx - 1) * (rng.uniform(0.35, 0.5) + rng.uniform(0.04, 0.1) * torch.cos(s) + 0.02 * torch.cos(3 * s))
    Ts, Tl = p["T_solidus"], p["T_liquidus"]
    T = torch.where(x < front, p["T_hot"] + (Tl - p["T_hot"]) * x / front,
                    Ts + (p["T_cold"] - Ts) * (x - front) / (nx - 1 - front))
    fl = ((front - x) / 4 + 0.5).clamp(0, 1)
    H = c.c_ps * T.clamp(max=Ts) + fl * (c.H_fl - c.H_fs) + (T - Tl).clamp(min=0)
    T, fl = c.state_of(H)
    Tm = T + 0.01 * torch.sin(math.pi * x / (nx - 1)) * (1 + 0.3 * torch.cos(2 * s + rng.uniform(0, 6)))
    ux = uy = torch.zeros_like(T)
    f = None
    if p["flow"]:
        # a roll in the liquid: u from the stream function U L sin^2(pi x / front) sin^2(s)
        U = 2 * p["Da"] * p["Ra"] * p["k_f"] / p["L_char"]
        a, xi = U * front / math.pi, (x / front).clamp(max=1) * math.pi
        ux = a * torch.sin(xi) ** 2 * torch.sin(2 * s) * math.pi / ny
        uy = -U * torch.sin(2 * xi) * torch.sin(s) ** 2
        f = c.f_eq(torch.ones_like(T), ux, uy) - torch.tensor(W9, dtype=torch.float64, device="cuda")[:, None, None]
    real = torch.float64 if p["precision"] == 0 else torch.float32
    return tuple(None if a is None else a.to(real) for a in (f, c.g_eq(H, T, ux, uy), c.h_eq(Tm), Tm - T))


# ---------------------------------------------------------------------------
# The cases through the public entry points
# ---------------------------------------------------------------------------

class _State:
    pass


def prepare(case, seed):
    s = _State()
    s.case = case
    s.solvers = []
    for k, p in enumerate(_parameters(case, seed)):
        solver = lbm.Solver(p)
        solver.set_state(*[None if a is None else a.cpu().numpy() for a in _melting(p, seed + 1000 * k)])
        s.solvers.append(solver)
    s.batch = None
    if case["kind"] == "batch":
        s.batch = lbm.Batch(s.solvers, autotune=False).configure(128, case["map"])
    return s


def run(state):
    case, kind = state.case, SNAPSHOT.get(state.case["precision"])

    def snapshot(solver, names):
        f = solver.fields(names)
        return {k: v.to(kind) for k, v in f.items()} if kind else f

    if state.batch is not None:
        state.batch.step(case["steps"])
        return [snapshot(s, BATCH_FIELDS) for s in state.solvers]
    solver = state.solvers[0]
    solver.step(case["steps"])
    out = {}
    if case["diag"]:
        d = solver.diag()
        out["diag"] = [d["melt_frac"], d["enthalpy"], d["mass"]]
    out["fields"] = snapshot(solver, lbm.FIELDS)
    return out


def work(case):
    """A step's arithmetic needs about 220 operations for the flow lattice and, for each thermal lattice, 8 for each of
    its populations and 20 more; a pass reads the state once and writes it and the fields once."""
    q, flow, b = case.get("lattice", 5), case.get("flow", True), {"f64": 8, "f32": 4}.get(case["precision"], 2)
    wide = 8 if b == 8 else 4
    node = (9 * flow + 2 * (q - 1)) * b + 3 * wide   # moving populations, the two rest populations, the history
    if case["kind"] == "batch":
        nodes = sum(n * n for n in _sides(case))
        out = len(BATCH_FIELDS) * b
    else:
        nodes, out = case["nx"] * case["ny"], len(lbm.FIELDS) * b
    return {"bytes": nodes * (2 * node + out), "flops": nodes * case["steps"] * (220 * flow + 2 * (8 * q + 20))}


# ---------------------------------------------------------------------------
# The same pass in float64 with torch alone
# ---------------------------------------------------------------------------

M9 = ((1, 1, 1, 1, 1, 1, 1, 1, 1), (-4, -1, -1, -1, -1, 2, 2, 2, 2), (4, -2, -2, -2, -2, 1, 1, 1, 1),
      (0, 1, 0, -1, 0, 1, -1, -1, 1), (0, -2, 0, 2, 0, 1, -1, -1, 1), (0, 0, 1, 0, -1, 1, 1, -1, -1),
      (0, 0, -2, 0, 2, 1, 1, -1, -1), (0, 1, -1, 1, -1, 0, 0, 0, 0), (0, 0, 0, 0, 0, 1, -1, 1, -1))
M5 = ((1, 1, 1, 1, 1), (0, 1, 0, -1, 0), (0, 0, 1, 0, -1), (0, 1, 1, 1, 1), (0, 1, -1, 1, -1))


def _matrix(rows):
    m = torch.tensor(rows, dtype=torch.float64)
    return m.cuda(), torch.linalg.inv(m).cuda()


class _Reference:
    """The method of Sec. III in population space, node by node as the paper writes it."""

    def __init__(self, p, f, g, h, dT):
        self.p, self.c = p, _Constants(p)
        d = [None if a is None else a.to(torch.float64) for a in (f, g, h, dT)]
        self.f = None if d[0] is None else d[0] + torch.tensor(W9, dtype=torch.float64, device="cuda")[:, None, None]
        self.g, self.h, self.dT = d[1:]
        self.M9, self.M9i = _matrix(M9)
        self.M, self.Mi = _matrix(M9 if self.c.Q == 9 else M5)
        nx, ny = p["nx"], p["ny"]
        inner = (0 if p["periodic_y"] else 1, ny if p["periodic_y"] else ny - 1)
        ys = torch.arange(ny, device="cuda").clamp(inner[0], inner[1] - 1)
        xs = torch.arange(1, nx - 1, device="cuda")
        one = torch.ones_like
        # wall nodes (y, x), the nodes they take their state from, and the side whose temperature rule applies
        yy = torch.arange(ny, device="cuda")
        self.walls = [(0, (yy, one(yy) * 0), (ys, one(yy))), (1, (yy, one(yy) * (nx - 1)), (ys, one(yy) * (nx - 2)))]
        if not p["periodic_y"]:
            self.walls += [(2, (one(xs) * 0, xs), (one(xs), xs)),
                           (3, (one(xs) * (ny - 1), xs), (one(xs) * (ny - 2), xs))]

    def macro(self):
        """Streams, applies Eq. 52 on the walls, and returns the state of every node."""
        c, p = self.c, self.p

        def stream(a):
            return torch.stack([a[i].roll((EY[i], EX[i]), (0, 1)) for i in range(a.shape[0])])

        fp, g, h = None if self.f is None else stream(self.f), stream(self.g), stream(self.h)

        def thermal(g, h):
            H = g.sum(0)
            return (H, *c.state_of(H), h.sum(0))

        def velocity(fp, T, fl):
            rho = fp.sum(0)
            G = c.gbeta * (T - p["T_ref0"]) * fl
            vx = fl * (fp[1] - fp[3] + fp[5] - fp[6] - fp[7] + fp[8]) / rho
            vy = fl * (fp[2] - fp[4] + fp[5] + fp[6] - fp[7] - fp[8]) / rho + 0.5 * c.phi * G
            l0 = 0.5 * (1 + 0.5 * c.phi * c.nu * p["J"] / c.K)
            l1 = 0.5 * c.phi * p["F_phi"] / math.sqrt(c.K)
            den = l0 + torch.sqrt(l0 * l0 + l1 * torch.sqrt(vx * vx + vy * vy))
            return rho, G, vx / den, vy / den

        H, T, fl, Tm = thermal(g, h)
        rho, G, ux, uy = velocity(fp, T, fl) if fp is not None else (torch.ones_like(T),) + (torch.zeros_like(T),) * 3
        new = []
        for side, at, src in self.walls:
            a = [None if v is None else v[(..., *src)] for v in (fp, g, h, H, T, Tm, rho, ux, uy)]
            fs, gs, hs, Hs, Ts, Tms, rs, us, vs = a
            if p["wall_kind"][side] == 0:
                Tb = torch.full_like(Ts, p["wall_T"][side])
                Hb, Tmb = torch.full_like(Ts, c.enthalpy(p["wall_T"][side])), Tb
            else:
                Hb, Tb, Tmb = Hs, Ts, Tms
            z = torch.zeros_like(Ts)
            fw = None if fs is None else fs + c.f_eq(rs, z, z) - c.f_eq(rs, us, vs)
            new.append((at, fw, gs + c.g_eq(Hb, Tb, z, z) - c.g_eq(Hs, Ts, us, vs), hs + c.h_eq(Tmb) - c.h_eq(Tms)))
        for at, fw, gw, hw in new:
            g[(..., *at)], h[(..., *at)] = gw, hw
            H[at], T[at], fl[at], Tm[at] = thermal(gw, hw)
            ux[at], uy[at] = 0.0, 0.0
            if fw is not None:
                fp[(..., *at)] = fw
                rho[at] = fw.sum(0)
                G[at] = c.gbeta * (T[at] - p["T_ref0"]) * fl[at]
        return fp, g, h, H, T, fl, Tm, rho, G, ux, uy

    def step(self):
        c, p, phi = self.c, self.p, self.c.phi
        fp, g, h, H, T, fl, Tm, rho, G, ux, uy = self.macro()
        if fp is not None:
            um = torch.sqrt(ux * ux + uy * uy)
            drag = phi * c.nu / c.K + phi * p["F_phi"] / math.sqrt(c.K) * um
            Fx, Fy = -drag * ux, -drag * uy + phi * G
            z = torch.zeros_like(T)
            m = torch.tensordot(self.M9, fl * fp + (1 - fl) * c.f_eq(rho, z, z), 1)
            me = torch.tensordot(self.M9, c.f_eq(rho, ux, uy), 1)
            uF, q = ux * Fx + uy * Fy, rho / phi
            S = torch.stack([z, 6 * q * uF, -6 * q * uF, rho * Fx, -rho * Fx, rho * Fy, -rho * Fy,
                             2 * q * (ux * Fx - uy * Fy), q * (ux * Fy + uy * Fx)])
            sv = 1 / (0.5 + 3 * c.nu * p["J"])
            s = torch.tensor([1, 1.1, 1.1, 1, 1.2, 1, 1.2, sv, sv], dtype=torch.float64, device="cuda")[:, None, None]
            self.f = torch.tensordot(self.M9i, m - s * (m - me) + (1 - 0.5 * s) * S, 1)
        dT = Tm - T
        X = c.h_v * (1.5 * dT - 0.5 * self.dT)
        self.dT = dT
        k = fl * p["k_f"] + (1 - fl) * c.k_s
        za = 1 / (0.5 + k / (p["cfref_over_cpl"] * c.cs2))
        a, one = c.eta, torch.ones_like(za)
        z0 = torch.zeros_like(ux)
        if c.Q == 9:
            rates = [one, 2 - za, 2 - za, za, za, za, za, 1.2 * one, 1.2 * one]
            eta, way = [1, 1.1, 1.1, a, a, a, a, 1.2, 1.2], [1, -2, 1, 0, 0, 0, 0, 0, 0]
        else:
            rates = [one, za, za, 2 - za, 1.2 * one]
            eta, way = [1, a, a, 1.1, 1.2], [1, 0, 0, p["varpi"], 0]
        way = torch.tensor(way, dtype=torch.float64, device="cuda")[:, None, None]
        eta = torch.tensor(eta, dtype=torch.float64, device="cuda")[:, None, None]
        jx, jy = T * ux / phi, T * uy / phi   # moments of Eqs. 34, 45 (B2, B4)
        if c.Q == 9:
            e, d = p["cfref_over_cpl"] * T, p["cmref_over_cpm"] * Tm
            ng = torch.stack([H, -4 * H + 2 * e, 4 * H - 3 * e, jx, -jx, jy, -jy, z0, z0])
            nh = torch.stack([Tm, -4 * Tm + 2 * d, 4 * Tm - 3 * d] + [z0] * 6)
        else:
            ng = torch.stack([H, jx, jy, p["varpi"] * p["cfref_over_cpl"] * T, z0])
            nh = torch.stack([Tm, z0, z0, p["varpi"] * p["cmref_over_cpm"] * Tm, z0])
        n = torch.tensordot(self.M, g, 1)
        self.g = torch.tensordot(self.Mi, n - torch.stack(rates) * (n - ng) + X / phi * way, 1)
        n = torch.tensordot(self.M, h, 1)
        self.h = torch.tensordot(self.Mi, n - eta * (n - nh) - X / ((1 - phi) * c.rho_m) * way, 1)


def exact(case, seed):
    out = []
    for k, p in enumerate(_parameters(case, seed)):
        r = _Reference(p, *_melting(p, seed + 1000 * k))
        for _ in range(case["steps"]):
            r.step()
        _, _, _, H, T, fl, Tm, rho, _, ux, uy = r.macro()
        fields = dict(T_f=T, T_s=Tm, f_l=fl, u_x=ux, u_y=uy, rho=rho, H_f=H)
        if case["kind"] == "batch":
            out.append({name: fields[name] for name in BATCH_FIELDS})
            continue
        res = {}
        if case["diag"]:
            phi = p["porosity"]
            res["diag"] = [float(fl.mean()), float((phi * H + (1 - phi) * r.c.rho_m * Tm).sum()), float(rho.sum())]
        res["fields"] = fields
        return res
    return out
