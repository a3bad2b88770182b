"""Measured cases of the pipe-flow lattice Boltzmann library.

Every case is one piece of work that a program of this library does over and over: advance
a pipe by a chunk of steps and look at its fields (run_pipe.py, bench.py), advance an
ensemble, evaluate an objective with its gradients (optimisation), or take the diagnostics
of a state.  Sizes are those of paper_2405_12082_gb300/workloads.py, of the tests and of
bench.py; `draw` spreads the same kinds over the ranges between them.

`exact` is the method in plain torch FP64 (literal two-buffer stream and collide), written
from the equations.  FP32 and 16-bit runs hand their FP64 diagnostics back in the precision
their populations carry.
"""
import math

import torch

from paper_2405_12082_gb300 import lbm
from paper_2405_12082_gb300 import workloads as Wk

# the paper's relaxation rate (tau = 0.5096) and velocity noise: stable for runs of any length
OMEGA, NOISE, U_STAR = Wk.C4["omega"], Wk.C4["noise"], Wk.C4["u_star"]
STORAGE = {"f64": torch.float64, "f32": torch.float32, "f16s": torch.float16, "bf16": torch.bfloat16}
FIELD = {"f64": torch.float64, "f32": torch.float32}          # what lbm_moments writes (float32 for 16-bit storage)


def _pipe(name, cfg, **more):
    case = dict(name=name, kind="step", geometry="pipe", nx=cfg["nx"], ny=cfg["ny"], nz=cfg["nz"], R=cfg["R"],
                precision="f32", wall="halfway", model="mrt", equilibrium="hermite6", steps=20, stats_every=0,
                modes=False, flow="turbulent", omega=OMEGA)
    case.update(more)
    return case


def listed():
    return [
        # the laminar FP64 verification pipe (full-way walls), in chunks of 100 steps: many tiny launches
        _pipe("laminar_f64_fullway", Wk.C1, precision="f64", wall="fullway", steps=100, flow="laminar", omega=1.25),
        # a small FP32 laminar pipe as the tests and first experiments use it
        _pipe("laminar_f32_small", dict(nx=28, ny=28, nz=64, R=11.5), steps=100, flow="laminar", omega=1.25),
        # the R = 48 pipe: 100 steps with one statistics sample, then the ring analysis (bench.py's step)
        _pipe("turbulent_f32_r48", Wk.C2, steps=100, stats_every=100, modes=True),
        # the paper's 300 x 300 x 600 production run: ring analysis every 20 steps (run_pipe.py)
        _pipe("paper_f32", Wk.C_PAPER, steps=20, modes=True),
        # the R = 96 pipe with the paper's own wall rule (run_pipe.py --wall bouzidi)
        _pipe("large_f32_bouzidi_r96", Wk.C3, steps=20, wall="bouzidi", modes=True),
        # throughput storage: the R = 96 pipe in scaled half, the R = 48 pipe in bfloat16
        _pipe("large_f16s_r96", Wk.C3, steps=40, precision="f16s"),
        _pipe("turbulent_bf16_r48", Wk.C2, steps=100, precision="bf16"),
        # FP64 storage as the reference of a precision study (precision_study.py)
        _pipe("precision_f64_r48", Wk.C2, steps=10, precision="f64", stats_every=10),
        # collision ablation (single relaxation time, second-order equilibrium) on the R = 48 pipe
        _pipe("ablation_bgk_o2_r48", Wk.C2, steps=50, model="bgk", equilibrium="order2"),
        # 16 pipes of four radii advanced together in graph chunks of 100 steps
        dict(name="ensemble_f32_16", kind="ensemble", members=16, nz=256, radii="16,20,24,32", precision="f32",
             wall="halfway", steps=100, graph=100),
        # objective and gradients of the adjoint pipe over its full horizon
        dict(name="adjoint_f32_r24", kind="adjoint", nx=52, ny=52, nz=256, R=24.0, precision="f32", T=2000, every=0,
             objective="ubulk", omega=1.25),
        # diagnostics of a state of the R = 96 pipe: fields, mass and momentum, rings at three radii
        dict(name="analysis_f32_r96", kind="analysis", nx=196, ny=196, nz=1152, R=96.0, precision="f32",
             wall="halfway", omega=OMEGA, rings="0.6,0.78,0.9", n_sections=16, n_modes=32),
    ]


def _log_uniform(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["step"] * 7 + ["ensemble", "adjoint", "adjoint", "analysis"])
    if kind == "ensemble":
        radii = sorted(rng.sample([12, 16, 18, 20, 24, 28, 32, 40], rng.randint(1, 4)))
        return dict(kind=kind, members=rng.randint(2, 24), nz=rng.randint(48, 256), radii=",".join(map(str, radii)),
                    precision=rng.choice(["f32", "f32", "f16s"]), wall=rng.choice(["halfway", "bouzidi"]),
                    steps=100, graph=rng.choice([0, 20, 50, 100]))
    if kind == "adjoint":
        R = round(_log_uniform(rng, 6.0, 24.0), 2)
        side = math.ceil(2 * R) + rng.randint(2, 5)
        return dict(kind=kind, nx=side, ny=side + rng.randint(0, 3), nz=rng.randint(9, 128), R=R,
                    precision=rng.choice(["f32", "f32", "f32", "f64"]) if R < 10 else "f32", T=rng.randint(20, 160),
                    every=rng.choice([0, 0, 13]), objective=rng.choice(["ubulk", "wss"]), omega=1.25)
    if kind == "analysis":
        R = round(_log_uniform(rng, 10.0, 96.0), 2)
        side = math.ceil(2 * R) + rng.randint(3, 6)
        return dict(kind=kind, nx=side, ny=side, nz=int(_log_uniform(rng, 32, 1000)), R=R,
                    precision=rng.choice(["f32", "f32", "f16s"]), wall=rng.choice(["halfway", "bouzidi", "fullway"]),
                    omega=OMEGA, rings=rng.choice(["0.78", "0.5,0.78"]), n_sections=rng.choice([4, 16]), n_modes=32)
    precision = rng.choice(["f32", "f32", "f32", "f16s", "bf16", "f64"])
    wall = rng.choice(["halfway", "halfway", "bouzidi", "fullway"])
    model, equilibrium = "mrt", "hermite6"
    if precision in ("f32", "f64") and rng.random() < 0.2:
        model, equilibrium = rng.choice([("bgk", "hermite6"), ("bgk", "order2"), ("mrt", "order2")])
    if rng.random() < 0.12:                                   # periodic box, every cell fluid
        side = int(_log_uniform(rng, 16, 64 if precision == "f64" else 200))
        c = dict(geometry="box", nx=side, ny=side + rng.randint(0, 5), nz=side + rng.randint(0, 9), R=0.0)
        wall = "halfway"
    else:
        R = round(_log_uniform(rng, 6.0, 40.0 if precision == "f64" else 110.0), 2)
        side = math.ceil(2 * R) + rng.randint(2, 5)
        c = dict(geometry="pipe", nx=side, ny=side + rng.randint(0, 3), R=R,
                 nz=int(_log_uniform(rng, 24, 320 if precision == "f64" else 700)))
    cells = c["nx"] * c["ny"] * c["nz"]
    budget = 2.5e7 if precision == "f64" else 5e8             # cell updates of a pass
    steps = max(4, min(rng.choice([20, 21, 50, 100]), int(budget / cells)))
    laminar = c["nx"] < 40 or c["geometry"] == "box"
    return dict(kind="step", precision=precision, wall=wall, model=model, equilibrium=equilibrium, steps=steps,
                stats_every=rng.choice([0, 0, 10, 100]), modes=c["geometry"] == "pipe" and R > 10 and rng.random() < 0.5,
                flow="laminar" if laminar else "turbulent", omega=1.25 if laminar else OMEGA, **c)


# ---- set-up ---------------------------------------------------------------------------------
def _fluid(case, device="cuda"):
    """(ny, nx) mask: distance to the axis below R; a box is fluid everywhere."""
    if case.get("geometry", "pipe") == "box":
        return torch.ones((case["ny"], case["nx"]), dtype=torch.bool, device=device)
    x = torch.arange(case["nx"], dtype=torch.float64, device=device) - (case["nx"] - 1) / 2
    y = torch.arange(case["ny"], dtype=torch.float64, device=device) - (case["ny"] - 1) / 2
    return x[None, :] ** 2 + y[:, None] ** 2 < case["R"] ** 2


def _is_turbulent(case):
    return case.get("flow", "turbulent") == "turbulent" and case["kind"] != "adjoint"


def _drive(case):
    """Constant axial acceleration: 2 u*^2 / R of the turbulent pipes, 1e-6 of the laminar ones."""
    if case["kind"] == "adjoint":
        return 0.0
    return 2.0 * U_STAR ** 2 / case["R"] if _is_turbulent(case) else 1e-6


def _trigger(case):
    """The four-mode trigger force of the turbulent pipes (active throughout)."""
    if not _is_turbulent(case) or case.get("geometry", "pipe") == "box":
        return None
    R = case["R"]
    return Wk.trigger_dict(h=_drive(case), R=R, nz=case["nz"], period=0.052 * R / U_STAR,
                           modes=[(m, 0.25, case.get("phase", 0.0)) for m in range(1, 5)], t_end=2 ** 40)


def _fields(case, seed):
    """rho and u (FP64, device) of the initial state: the mean profile with noise, or a slow laminar one."""
    gen = torch.Generator(device="cuda").manual_seed(int(seed))
    nz, ny, nx = case["nz"], case["ny"], case["nx"]
    u = torch.randn((3, nz, ny, nx), generator=gen, device="cuda", dtype=torch.float32).double()
    if _is_turbulent(case):
        u *= NOISE
        nu = (1.0 / case["omega"] - 0.5) / 3.0
        x = torch.arange(nx, dtype=torch.float64, device="cuda") - (nx - 1) / 2
        y = torch.arange(ny, dtype=torch.float64, device="cuda") - (ny - 1) / 2
        dplus = (case["R"] - (x[None, :] ** 2 + y[:, None] ** 2).sqrt()).clamp(min=1e-9) * U_STAR / nu
        u[2] += U_STAR * torch.where(dplus <= 10.8, dplus, dplus.log() / 0.4 + 5.0)
    else:
        u *= 1e-3
        u[2] += 0.01
    rho = 1.0 + 1e-3 * torch.randn((nz, ny, nx), generator=gen, device="cuda", dtype=torch.float32).double()
    return rho.contiguous(), u.contiguous()


def _grid(case):
    return lbm.make_grid(case["nx"], case["ny"], case["nz"], case["R"], geometry=case.get("geometry", "pipe"),
                         precision=case["precision"], wall=case.get("wall", "halfway"))


def _force(case):
    return lbm.make_force(g=(0.0, 0.0, _drive(case)), trigger=_trigger(case))


def _members(case, seed):
    """The pipes of an ensemble: radii drawn from the list, box 2R + 4, a trigger phase each."""
    gen = torch.Generator().manual_seed(12345)                # the geometry is the case's, not the seed's
    radii = [int(r) for r in case["radii"].split(",")]
    pick = torch.randint(len(radii), (case["members"],), generator=gen).tolist()
    return [dict(kind="step", geometry="pipe", nx=2 * radii[k] + 4, ny=2 * radii[k] + 4, nz=case["nz"],
                 R=float(radii[k]), precision=case["precision"], wall=case["wall"], omega=OMEGA, flow="turbulent",
                 model="mrt", equilibrium="hermite6", steps=case["steps"], phase=2 * math.pi * m / case["members"],
                 member_seed=int(seed) * 64 + m) for m, k in enumerate(pick)]


def _rings(case):
    """Rings of the analysis; as many samples as the smallest power of two above the circumference."""
    rings = [float(r) for r in case.get("rings", "0.78").split(",")]
    n_theta = 1 << max(3, math.ceil(math.log2(2 * math.pi * max(rings) * case["R"])))
    return rings, n_theta, min(case.get("n_sections", 16), case["nz"]), min(case.get("n_modes", 32), n_theta - 1)


def _gz(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(int(seed) + 77)
    r = torch.rand((case["nz"], case["ny"], case["nx"]), generator=gen, device="cuda", dtype=torch.float32)
    return (1e-6 * (0.7 + 0.6 * r)).to(FIELD[case["precision"]]).contiguous()


def prepare(case, seed):
    s = {"case": case}
    if case["kind"] == "ensemble":
        members = _members(case, seed)
        s["members"] = members
        L = lbm.Lattice(None, None, ensemble=([_grid(m) for m in members], [lbm.lbm_relax(OMEGA) for _ in members],
                                              [_force(m) for m in members]))
        for k, m in enumerate(members):
            L.select(k)
            lbm.lbm_init_fields(L.ctx, *_fields(m, m["member_seed"]))
        torch.cuda.synchronize()
        if case["graph"]:
            lbm.lbm_set_graph(L.ctx, case["graph"])
    else:
        L = lbm.Lattice(_grid(case), lbm.lbm_relax(case["omega"]), _force(case))
        if case.get("model", "mrt") != "mrt" or case.get("equilibrium", "hermite6") != "hermite6":
            lbm.lbm_set_collision(L.ctx, case["model"], case["equilibrium"])
        rho, u = _fields(case, seed)
        lbm.lbm_init_fields(L.ctx, rho, u)
        torch.cuda.synchronize()
        del rho, u
        if case.get("stats_every"):
            lbm.lbm_stats_enable(L.ctx, case["stats_every"])
    s["L"] = L
    if case["kind"] == "adjoint":
        s["gz"] = _gz(case, seed).requires_grad_(True)
        s["omega"] = torch.tensor(case["omega"], dtype=FIELD[case["precision"]], requires_grad=True)
    elif case["kind"] in ("step", "ensemble"):
        dt = STORAGE[case["precision"]]
        s["raw"] = torch.empty(L.info()["population_bytes"] // torch.empty(0, dtype=dt).element_size(), dtype=dt,
                               device="cuda")
    if case.get("modes") or case["kind"] == "analysis":
        rings, n_theta, n_sections, n_modes = _rings(case)
        s["cfg"] = lbm.make_modes_cfg(n_sections, rings, n_theta, n_modes)
        s["E"] = torch.empty((n_sections, len(rings), n_modes + 1), dtype=torch.float64, device="cuda")
    return s


# ---- one pass -------------------------------------------------------------------------------
def _moments(L, case):
    """rho and u; a 16-bit run keeps them in its storage type."""
    rho, u = L.moments()
    return (rho, u) if case["precision"] in FIELD else (rho.to(STORAGE[case["precision"]]), u.to(STORAGE[case["precision"]]))


def _spectrum(s):
    lbm.lbm_modes(s["L"].ctx, s["cfg"], s["E"])
    p = s["case"]["precision"]
    return s["E"].to(torch.float64 if p == "f64" else torch.float32 if p == "f32" else torch.bfloat16)


def run(s):
    case, L = s["case"], s["L"]
    if case["kind"] == "adjoint":
        s["gz"].grad = s["omega"].grad = None
        J = lbm.pipe_objective(L, s["gz"], s["omega"], case["T"], case["objective"], case["every"])
        J.backward()
        rho, u = L.moments()
        return {"J": J.detach().to(s["gz"].dtype), "dgz": s["gz"].grad, "domega": s["omega"].grad, "rho": rho, "u": u}
    if case["kind"] == "analysis":
        rho, u = _moments(L, case)
        E = _spectrum(s)
        sums = lbm.lbm_reduce(L.ctx)
        return {"rho": rho, "u": u, "E": E, "sums": sums if case["precision"] in FIELD else sums[4]}
    L.step(case["steps"])
    raw = s["raw"]
    lbm.lbm_get_raw(L.ctx, raw, raw.numel() * raw.element_size())
    out = {"raw": raw}
    if case["kind"] == "ensemble":
        for k in range(case["members"]):
            L.select(k)
            out["rho%d" % k], out["u%d" % k] = _moments(L, case)
        return out
    out["rho"], out["u"] = _moments(L, case)
    if case["modes"]:
        out["E"] = _spectrum(s)
    return out


# ---- what a pass cannot do without ----------------------------------------------------------
def work(case):
    es = {"f64": 8, "f32": 4, "f16s": 2, "bf16": 2}[case["precision"]]
    fs = 8 if case["precision"] == "f64" else 4
    if case["kind"] == "ensemble":
        cells = [(int(_fluid(m, "cpu").sum()) * m["nz"], m["nx"] * m["ny"] * m["nz"]) for m in _members(case, 0)]
        fluid, dense = sum(c[0] for c in cells), sum(c[1] for c in cells)
    else:
        fluid = int(_fluid(case, "cpu").sum()) * case["nz"]
        dense = case["nx"] * case["ny"] * case["nz"]
    fields = 27 * es * fluid + 4 * fs * dense                 # populations read, rho and u written
    if case["kind"] == "analysis":
        return {"bytes": fields, "flops": 100 * fluid}
    if case["kind"] == "adjoint":
        # a forward step (27 populations in and out) and a reverse step (27 adjoint values in and
        # out, g_z, its gradient); states in between may be kept or recomputed
        return {"bytes": case["T"] * fluid * (4 * 27 * es + 3 * fs) + fields, "flops": case["T"] * fluid * 1000}
    out = fields + (2 * 27 * es * fluid)                      # the copy of the state handed back
    return {"bytes": case["steps"] * fluid * 2 * 27 * es + out, "flops": case["steps"] * fluid * 320}


# ---- the method in FP64 ---------------------------------------------------------------------
CX = (0, 1, -1, 0, 0, 0, 0, 1, -1, 1, -1, 1, -1, 1, -1, 0, 0, 0, 0, 1, -1, 1, -1, 1, -1, 1, -1)
CY = (0, 0, 0, 1, -1, 0, 0, 1, 1, -1, -1, 0, 0, 0, 0, 1, -1, 1, -1, 1, 1, -1, -1, 1, 1, -1, -1)
CZ = (0, 0, 0, 0, 0, 1, -1, 0, 0, 0, 0, 1, 1, -1, -1, 1, 1, -1, -1, 1, 1, 1, 1, -1, -1, -1, -1)
W = [8 / 27 if i == 0 else 2 / 27 if i < 7 else 1 / 54 if i < 19 else 1 / 216 for i in range(27)]
C3 = list(zip(CX, CY, CZ))
OPP = [C3.index((-x, -y, -z)) for x, y, z in C3]


def _moment_rows(x, y, z):
    """The moment basis at one velocity."""
    x2, y2, z2 = x * x, y * y, z * z
    return [1, x, y, z, x * y, x * z, y * z, x2 - y2, x2 - z2, x2 + y2 + z2, x * (y2 + z2), y * (x2 + z2),
            z * (x2 + y2), x * (y2 - z2), y * (x2 - z2), z * (x2 - y2), x * y * z, x2 * y2 + x2 * z2 + y2 * z2,
            x2 * y2 + x2 * z2 - y2 * z2, x2 * y2 - x2 * z2, x2 * y * z, x * y2 * z, x * y * z2, x * y2 * z2,
            x2 * y * z2, x2 * y2 * z, x2 * y2 * z2]


_MT = torch.tensor([_moment_rows(*c) for c in C3], dtype=torch.float64).T.contiguous()     # m = _MT f
_MT_INV = torch.linalg.inv(_MT)


class _Exact:
    """Literal stream and collide of one pipe or box, FP64."""

    def __init__(self, case):
        self.case = case
        nz, ny, nx = case["nz"], case["ny"], case["nx"]
        col = _fluid(case)
        self.fluid = col.expand(nz, ny, nx)
        self.wall = case.get("wall", "halfway") if case.get("geometry", "pipe") == "pipe" else "box"
        # is x - c_i fluid (periodic)
        self.src = [torch.roll(col, shifts=(CY[i], CX[i]), dims=(0, 1)) for i in range(27)]
        self.col = col
        self.table = None
        self.x = torch.arange(nx, dtype=torch.float64, device="cuda") - (nx - 1) / 2
        self.y = torch.arange(ny, dtype=torch.float64, device="cuda") - (ny - 1) / 2
        self.tr = _trigger(case)
        if self.tr:
            self._trigger_columns()
        if self.wall == "bouzidi":
            self.links = [self._bouzidi(j) for j in range(27)]

    def _trigger_columns(self):
        """The trigger force is sin(2 pi t / T) times these columns times cos (x, y) or sin (z) of kz 2 pi z / L."""
        tr, R, L = self.tr, self.case["R"], self.case["nz"]
        X, Y = self.x[None, :].expand(len(self.y), -1), self.y[:, None].expand(-1, len(self.x))
        r, th = (X * X + Y * Y).sqrt(), torch.atan2(Y, X)
        band = (r >= R - tr["l0"] - tr["l"]) & (r <= R - tr["l0"]) & (r > 0)
        arg, rs = 2 * math.pi * (R - r - tr["l0"]) / tr["l"], r.clamp(min=1e-12)
        Fr, Ft, Fz = torch.zeros_like(r), torch.zeros_like(r), torch.zeros_like(r)
        for kt, weight, phase in tr["modes"]:
            A, ang = tr["h"] * tr["A0"] * weight, kt * th + phase
            Fr -= A * tr["kappa"] * (R / rs) * (tr["kz"] * tr["l"] / L) * (1 - arg.cos()) * ang.cos()
            Ft += A * (1 - tr["kappa"]) * (tr["kz"] / kt) * (2 * math.pi * R / L) * arg.sin() * ang.sin()
            Fz -= A * (R / rs) * arg.sin() * ang.cos()
        zero = torch.zeros_like(r)
        self.trig = [torch.where(band, f, zero) for f in (Fr * th.cos() - Ft * th.sin(), Fr * th.sin() + Ft * th.cos(), Fz)]
        z = torch.arange(L, dtype=torch.float64, device="cuda") * (2 * math.pi * tr["kz"] / L)
        self.zc, self.zs = z.cos()[:, None, None], z.sin()[:, None, None]

    def _bouzidi(self, j):
        """A, B, C of the reflection of direction j at a wall link of Bouzidi's interpolation."""
        cx, cy = CX[j], CY[j]
        if cx == 0 and cy == 0:
            return None
        a = float(cx * cx + cy * cy)
        px, py = self.x[None, :], self.y[:, None]
        b, c = px * cx + py * cy, px * px + py * py - self.case["R"] ** 2
        d = ((-b + (b * b - a * c).clamp(min=0).sqrt()) / a).clamp(min=1e-12)
        ff = torch.roll(self.col, shifts=(cy, cx), dims=(0, 1))
        one, zero = torch.ones_like(d), torch.zeros_like(d)
        near = d < 0.5
        return (torch.where(near, torch.where(ff, 2 * d, one), 1 / (2 * d)),
                torch.where(near, zero, (2 * d - 1) / (2 * d)), torch.where(near & ff, 1 - 2 * d, zero))

    def accel(self, t, gz=None):
        g = [0.0, 0.0, _drive(self.case)]
        if gz is not None:
            g[2] = g[2] + gz
        if self.tr:
            st = math.sin(2 * math.pi * t / self.tr["period"])
            g = [g[0] + st * self.zc * self.trig[0], g[1] + st * self.zc * self.trig[1], g[2] + st * self.zs * self.trig[2]]
        return g

    def start(self, rho, u):
        """Equilibrium of the model at (rho, u) on fluid cells, rest elsewhere."""
        return torch.stack([torch.where(self.fluid, q, torch.full_like(q, W[i]))
                            for i, q in enumerate(self._populations(rho, u, [0.0, 0.0, 0.0], force=False))])

    def _populations(self, rho, u, g, force=True):
        """Yields f^eq_i, or with force (f^eq_i, g . grad_u f^eq_i)."""
        if self.case.get("equilibrium", "hermite6") == "order2":
            uu = u[0] * u[0] + u[1] * u[1] + u[2] * u[2]
            ug = u[0] * g[0] + u[1] * g[1] + u[2] * g[2]
            for i, c in enumerate(C3):
                cu = c[0] * u[0] + c[1] * u[1] + c[2] * u[2]
                cg = c[0] * g[0] + c[1] * g[1] + c[2] * g[2]
                eq = W[i] * rho * (1 + 3 * cu + 4.5 * cu * cu - 1.5 * uu)
                yield (eq, W[i] * rho * (3 * (cg - ug) + 9 * cu * cg)) if force else eq
            return
        p, q = [], []                                         # psi and g psi' of every axis at c = -1, 0, 1
        for k in range(3):
            p.append([1 - 3 * u[k] + 3 * u[k] * u[k], 1 - 1.5 * u[k] * u[k], 1 + 3 * u[k] + 3 * u[k] * u[k]])
            q.append([g[k] * (6 * u[k] - 3), g[k] * (-3 * u[k]), g[k] * (6 * u[k] + 3)])
        for i, (a, b, c) in enumerate(C3):
            a, b, c = a + 1, b + 1, c + 1
            pxy = p[0][a] * p[1][b]
            eq = W[i] * rho * pxy * p[2][c]
            if force:
                yield eq, W[i] * rho * ((q[0][a] * p[1][b] + p[0][a] * q[1][b]) * p[2][c] + pxy * q[2][c])
            else:
                yield eq

    def macro(self, f, g):
        rho = f.sum(0)
        u = []
        for k, c in enumerate((CX, CY, CZ)):
            j = 0
            for i in range(27):
                if c[i]:
                    j = j + c[i] * f[i]
            u.append(j / rho + 0.5 * g[k])
        return rho, u

    def collide(self, f, g, omega):
        rho, u = self.macro(f, g)
        if self.case.get("model", "mrt") == "bgk":
            return torch.stack([torch.where(self.fluid, eq + 0.5 * F + (1 - omega) * (f[i] - eq + 0.5 * F), f[i])
                                for i, (eq, F) in enumerate(self._populations(rho, u, g))])
        s = [0] * 5                                           # non-equilibrium moments 4..8
        for i, (eq, F) in enumerate(self._populations(rho, u, g)):
            n = f[i] - eq + 0.5 * F
            for k in range(5):
                m = float(_MT[4 + k, i])
                if m:
                    s[k] = s[k] + m * n
        out = []
        for i, (eq, F) in enumerate(self._populations(rho, u, g)):
            q = eq + 0.5 * F
            for k in range(5):
                w = float(_MT_INV[i, 4 + k])
                if abs(w) > 1e-12:
                    q = q + ((1 - omega) * w) * s[k]
            out.append(torch.where(self.fluid, q, f[i]))
        return torch.stack(out)

    def step(self, f, t, omega=None, gz=None):
        """f after one step, and the post-collision populations."""
        fs = self.collide(f, self.accel(t, gz), self.case["omega"] if omega is None else omega)
        if self.wall == "fullway":
            fs = torch.where(self.fluid, fs, f[OPP])
        new = []
        for i, c in enumerate(C3):
            q = torch.roll(fs[i], shifts=(c[2], c[1], c[0]), dims=(0, 1, 2))
            if self.wall in ("halfway", "bouzidi") and (c[0] or c[1]):
                j = OPP[i]
                back = fs[j]
                if self.wall == "bouzidi":
                    A, B, C = self.links[j]
                    cj = C3[j]
                    back = A * fs[j] + B * fs[i] + C * torch.roll(fs[j], shifts=(cj[2], cj[1], cj[0]), dims=(0, 1, 2))
                q = torch.where(self.src[i], q, back)
            if self.wall != "fullway":
                q = torch.where(self.fluid, q, f[i])
            new.append(q)
        return torch.stack(new), fs

    def moments(self, f, t, gz=None):
        rho, u = self.macro(f, self.accel(t, gz))
        zero = torch.zeros_like(rho)
        return torch.where(self.fluid, rho, zero), torch.stack([torch.where(self.fluid, q, zero) for q in u])

    def spectrum(self, uz):
        """|sum_n u_z exp(-i m theta_n)|^2 / N^2 on every ring, bilinear samples."""
        rings, N, ns, M = _rings(self.case)
        z = torch.tensor([s * self.case["nz"] // ns for s in range(ns)], device="cuda")
        th = torch.arange(N, dtype=torch.float64, device="cuda") * (2 * math.pi / N)
        ph = torch.outer(torch.arange(M + 1, dtype=torch.float64, device="cuda"), th)
        E = []
        for q in rings:
            px = (self.case["nx"] - 1) / 2 + q * self.case["R"] * th.cos()
            py = (self.case["ny"] - 1) / 2 + q * self.case["R"] * th.sin()
            i, j = px.floor().long(), py.floor().long()
            fx, fy = px - i, py - j
            v = uz[z]
            s = ((1 - fx) * (1 - fy) * v[:, j, i] + fx * (1 - fy) * v[:, j, i + 1] + (1 - fx) * fy * v[:, j + 1, i]
                 + fx * fy * v[:, j + 1, i + 1])
            E.append(((s @ ph.cos().T) ** 2 + (s @ ph.sin().T) ** 2) / N ** 2)
        return torch.stack(E, 1)


def _advance(case, seed):
    e = _Exact(case)
    f = e.start(*_fields(case, seed))
    for t in range(case["steps"]):
        f, _ = e.step(f, t)
    return e, f


def _exact_adjoint(case, seed):
    from torch.utils.checkpoint import checkpoint
    e = _Exact(case)
    rho0, u0 = _fields(case, seed)
    f = e.start(rho0, u0)
    gz = _gz(case, seed).double().requires_grad_(True)
    omega = torch.tensor(case["omega"], dtype=FIELD[case["precision"]]).double().cuda().requires_grad_(True)
    n, area = float(e.fluid.sum()), 2 * math.pi * case["R"] * case["nz"]

    def one(f, gz, omega):
        if case["objective"] == "ubulk":
            uz = e.macro(f, e.accel(0, gz))[1][2]
            return e.step(f, 0, omega, gz)[0], torch.where(e.fluid, uz, torch.zeros_like(uz)).sum() / n
        new, fs = e.step(f, 0, omega, gz)
        J = 0.0
        for i, c in enumerate(C3):
            if c[2] and (c[0] or c[1]):                       # links from fluid x into the wall
                J = J + 2 * c[2] * torch.where(e.col & ~e.src[OPP[i]], fs[i], torch.zeros_like(fs[i])).sum() / area
        return new, J

    J = 0.0
    for _ in range(case["T"]):
        f, a = checkpoint(one, f, gz, omega, use_reentrant=False)
        J = J + a / case["T"]
    J.backward()
    rho, u = e.moments(f.detach(), 0, gz.detach())
    return {"J": J.detach(), "dgz": gz.grad, "domega": omega.grad, "rho": rho, "u": u}


def exact(case, seed):
    if case["kind"] == "ensemble":
        members = _members(case, seed)
        out = {"raw": None}
        for k, m in enumerate(members):
            e, f = _advance(m, m["member_seed"])
            out["rho%d" % k], out["u%d" % k] = e.moments(f, m["steps"])
        return out
    cells = case["nx"] * case["ny"] * case["nz"]
    if case["kind"] == "adjoint":
        return _exact_adjoint(case, seed) if cells * case["T"] < 6e7 else None
    if case["kind"] == "analysis":
        e = _Exact(case)
        f = e.start(*_fields(case, seed))
        rho, u = e.moments(f, 0)
        d = [f[i] - W[i] for i in range(27)]
        sums = [float(torch.where(e.fluid, sum(d), torch.zeros_like(rho)).sum())]
        for c in (CX, CY, CZ):
            j = sum(c[i] * d[i] for i in range(27) if c[i])
            sums.append(float(torch.where(e.fluid, j, torch.zeros_like(j)).sum()))
        return {"rho": rho, "u": u, "E": e.spectrum(u[2]), "sums": sums + [0.0] if case["precision"] in FIELD else 0.0}
    if cells * case["steps"] > 2e9:
        return None
    e, f = _advance(case, seed)
    rho, u = e.moments(f, case["steps"])
    out = {"raw": None, "rho": rho, "u": u}
    if case["modes"]:
        out["E"] = e.spectrum(u[2])
    return out
