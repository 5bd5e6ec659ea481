"""The work this framework does for its users, as measurable cases.

Three kinds of call, each through the public binding
(``paper_1608_04118_gb300.ltne``):

- ``cavity``: one lattice of the differentially heated porous cavity.  A pass
  sets the initial fields from host arrays, advances ``steps`` time steps,
  reads the observables every ``every`` steps (a convergence monitor) and the
  fields at the end.
- ``sweep``: a parameter study, ``count`` independent cavities of uneven size
  advanced together by the batched form with the schedule its autotuner picks;
  a pass ends with every cavity's observables and fields.
- ``adjoint``: J = (Nu_f,hot + Nu_s,hot) / 2 after ``steps`` steps and its
  gradients with respect to the porosity field and to H.

Parameters are those of ``workloads.py`` and of the paper's Sec. 4; every
input that a user would bring (porosity, initial fields, the sweep's physical
parameters) is drawn from the seed.  ``exact`` restates the method in 64-bit
torch operations: moments by the printed matrices M and N, streaming by
rolls, walls by index lists, gradients by automatic differentiation.
"""
import math
import random

import numpy as np
import torch

from paper_1608_04118_gb300.ltne import LTNE_K_DARCY, LTNE_K_ERGUN, Batch, Cavity

# observables a monitor keeps (all but the step counter and the time)
OBS = ("Nu_f_hot", "Nu_s_hot", "Nu_f_cold", "Nu_s_cold", "mass", "energy", "max_u", "max_dT",
       "mean_Tf", "mean_Ts")
FIELDS = ("rho", "ux", "uy", "Tf", "Ts")
STORED = {"f64": 8, "f32": 4, "f16": 2, "bf16": 2}

PLAIN = dict(Ra=1e4, Da=1e-2, H=10.0, gamma_sf=1.0, ergun=False, T_hot=1.0, T_cold=0.0, T_ref=0.5,
             F_phi=-1.0, hv_local=False)
THROUGHPUT = dict(PLAIN, Ra=1e6, Da=1e-3, H=100.0, gamma_sf=10.0, ergun=True)
REDUCED = dict(PLAIN, Ra=1e6, Da=1e-2, H=1000.0)
GRADIENT = dict(PLAIN, Ra=1e5, Da=1e-3, H=50.0, ergun=True)
FOAM = dict(PLAIN, Ra=1e8, Da=1e-4, gamma_sf=1000.0, T_hot=11.0, T_cold=1.0, T_ref=1.0, F_phi=0.068,
            hv_local=True)


def _cavity(name, nx, ny, storage, steps, every, porosity, start, physics, **more):
    """porosity: "uniform" or "field"; start: "rest" (the temperatures only are
    given) or "fields" (all five)."""
    return dict(name=name, kind="cavity", nx=nx, ny=ny, storage=storage, steps=steps, every=every,
                porosity=porosity, start=start, **physics, **more)


def listed():
    return [
        # a small cavity run to convergence with a close monitor: the smallest
        # steps, launches and reads count
        _cavity("monitored 64x64 f32", 64, 64, "f32", 1000, 50, "uniform", "rest", PLAIN),
        # the same cavity as the double-precision reference run of a study
        _cavity("reference 64x64 f64", 64, 64, "f64", 500, 250, "uniform", "rest", PLAIN),
        # a user's own odd size, restarted from fields of another code
        _cavity("restart 131x97 f32", 131, 97, "f32", 400, 200, "field", "fields", THROUGHPUT),
        # the paper's metallic foam: local heat transfer coefficient of Eq. 52
        _cavity("foam 192x192 f32", 192, 192, "f32", 600, 300, "uniform", "rest", FOAM),
        # the forward run of the design problem
        _cavity("porous 256x256 f32", 256, 256, "f32", 600, 600, "field", "rest", GRADIENT),
        # a double-precision run of a mid-sized ragged cavity
        _cavity("reference 301x211 f64", 301, 211, "f64", 100, 100, "field", "fields", THROUGHPUT),
        # the throughput configuration at its two sizes
        _cavity("throughput 1024x1024 f32", 1024, 1024, "f32", 500, 250, "field", "rest", THROUGHPUT),
        _cavity("throughput 4096x4096 f32", 4096, 4096, "f32", 200, 200, "field", "rest", THROUGHPUT),
        # reduced storage: the large configuration, and a ragged porous one
        _cavity("reduced 8192x8192 f16", 8192, 8192, "f16", 80, 80, "uniform", "fields", REDUCED),
        _cavity("reduced 2049x1531 bf16", 2049, 1531, "bf16", 200, 200, "field", "fields", REDUCED),
        # a parameter study in the batched form
        dict(name="sweep of 12", kind="sweep", count=12, mix=3, steps=400),
        # a gradient of the design problem
        dict(GRADIENT, name="gradient 256x256 f32", kind="adjoint", nx=256, ny=256, storage="f32",
             steps=400),
    ]


def draw(rng):
    def spread(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["cavity"] * 6 + ["sweep"] + ["adjoint"] * 2)
    if kind == "sweep":
        return dict(kind="sweep", count=rng.randint(4, 12), mix=rng.randrange(1 << 20),
                    steps=spread(60, 400))
    if kind == "adjoint":
        nx, ny = spread(48, 400), spread(48, 400)
        return dict(GRADIENT, kind="adjoint", nx=nx, ny=ny, storage=rng.choice(["f32", "f32", "f64"]),
                    steps=max(40, min(400, int(1.5e7 / (nx * ny)))),
                    Ra=float("%.3g" % 10 ** rng.uniform(4, 6)))
    storage = rng.choice(["f32", "f32", "f32", "f16", "bf16", "f64"])
    side = spread(48, 600 if storage == "f64" else 4096)
    aspect = math.exp(rng.uniform(-0.5, 0.5))
    nx, ny = max(33, int(side * aspect)), max(33, int(side / aspect))
    if rng.random() < 0.5:  # half of the sizes are multiples of 32, as in the sweeps
        nx, ny = max(32, nx // 32 * 32), max(32, ny // 32 * 32)
    # reduced storage resolves a flow that is there, not the onset from rest
    start = "fields" if STORED[storage] == 2 else rng.choice(["rest", "rest", "fields"])
    work = 2e7 if storage == "f64" else 3e9  # node updates
    steps = max(40, min(800, int(work / (nx * ny))))
    physics = dict(rng.choice([PLAIN, THROUGHPUT, THROUGHPUT, REDUCED, GRADIENT, FOAM]))
    physics["Ra"] = float("%.3g" % (physics["Ra"] * 10 ** rng.uniform(-0.5, 0.5)))
    case = _cavity("", nx, ny, storage, steps, rng.choice([steps, max(1, steps // 3), 64]),
                   rng.choice(["uniform", "field", "field"]), start, physics)
    del case["name"]
    return case


# ---- inputs ------------------------------------------------------------------


def _sides(case):
    """The sizes of a sweep's cavities: sides 64, 96, ..., 512, aspect 1 or 2."""
    r = random.Random(case["mix"])
    out = []
    for _ in range(case["count"]):
        ny = r.randrange(64, 513, 32)
        out.append((ny * r.choice([1, 2]), ny))
    return out


def _sweep_params(case, seed):
    r = random.Random(seed)
    return [dict(nx=nx, ny=ny, Ra=10 ** r.uniform(3, 6), Da=10 ** r.uniform(-4, -1),
                 porosity=r.uniform(0.3, 0.9), H=10 ** r.uniform(0, 3),
                 gamma_sf=10 ** r.uniform(-1, 2), Pr=1.0, sigma=1.0, T_hot=1.0, T_cold=0.0, T_ref=0.5)
            for nx, ny in _sides(case)]


def _inputs(case, seed):
    """porosity and initial fields of a cavity as (ny, nx) float64 tensors on
    the GPU (absent ones take the framework's defaults): porosity independent
    per node, temperatures the conduction profile with smooth disturbances and
    some noise, and for a restart a cellular flow of the convection's speed."""
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    nx, ny = case["nx"], case["ny"]
    g = torch.Generator(device=dev).manual_seed(int(seed))
    r = random.Random(seed)

    def noise(lo, hi):
        return torch.empty((ny, nx), dtype=torch.float64, device=dev).uniform_(lo, hi, generator=g)

    out = {}
    foam = case["hv_local"]
    if case.get("porosity", "field") == "field":
        lo, hi = (0.7, 0.9) if foam else (0.4, 0.8) if case["kind"] == "adjoint" else (0.3, 0.9)
        out["porosity"] = noise(lo, hi)
    x = torch.linspace(0, 1, nx, dtype=torch.float64, device=dev)[None, :]
    y = torch.linspace(0, 1, ny, dtype=torch.float64, device=dev)[:, None]
    dT = case["T_hot"] - case["T_cold"]
    for key in ("T_f", "T_s"):
        wave = r.uniform(-0.1, 0.1) * torch.sin(math.pi * x) * torch.cos(math.pi * r.randint(1, 3) * y)
        t = (1 - x) + wave
        out[key] = case["T_cold"] + dT * t + 0.02 * dT * noise(-1, 1)
    if case.get("start") == "fields":
        u = 0.02 * r.uniform(0.5, 1.5)
        out["ux"] = u * torch.sin(math.pi * x) * torch.cos(math.pi * y) + 0.1 * u * noise(-1, 1)
        out["uy"] = -u * torch.cos(math.pi * x) * torch.sin(math.pi * y) + 0.1 * u * noise(-1, 1)
        out["rho"] = 1.0 + 0.002 * noise(-1, 1)
    return out


def _keywords(case):
    return dict(Ra=case["Ra"], Pr=1.0, Da=case["Da"], porosity=0.8 if case["hv_local"] else 0.6,
                H=case["H"], gamma_sf=case["gamma_sf"], sigma=1.0, T_hot=case["T_hot"],
                T_cold=case["T_cold"], T_ref=case["T_ref"], F_phi=case["F_phi"],
                hv_local=int(case["hv_local"]),
                permeability=LTNE_K_ERGUN if case["ergun"] else LTNE_K_DARCY)


def _host(t):
    """A page-locked host array with the tensor's values."""
    h = torch.empty(t.shape, dtype=torch.float64, pin_memory=True)
    h.copy_(t)
    return h.numpy()


def prepare(case, seed):
    if case["kind"] == "sweep":
        batch = Batch(_sweep_params(case, seed)).set_schedule(64, 4, 0, 2)
        return dict(case=case, batch=batch)
    field = case.get("porosity", "field") == "field"
    cav = Cavity(case["nx"], case["ny"], storage=case["storage"], porosity_field=int(field),
                 **_keywords(case))
    arrays = {k: _host(v) for k, v in _inputs(case, seed).items()}
    state = dict(case=case, cavity=cav, arrays=arrays, out=None)
    if case["kind"] == "cavity" and case["nx"] * case["ny"] > 1 << 19:
        # a program that reads large fields again and again keeps the arrays
        state["out"] = {k: torch.empty((case["ny"], case["nx"]), dtype=torch.float64,
                                       pin_memory=True).numpy() for k in FIELDS}
    return state


# ---- one pass ----------------------------------------------------------------


def run(state):
    case = state["case"]
    if case["kind"] == "sweep":
        b = state["batch"].set_fields().step(case["steps"])
        obs = b.observables()
        return dict(observables=np.array([[o[k] for k in OBS] for o in obs]),
                    fields=[b.fields(i) for i in range(b.count)])
    cav, arrays = state["cavity"], state["arrays"]
    if case["kind"] == "adjoint":
        J, g, dH = cav.adjoint(arrays["porosity"], case["steps"], T_f=arrays["T_f"], T_s=arrays["T_s"])
        return dict(J=J, dJ_dphi=g, dJ_dH=dH)
    cav.set_fields(**arrays)
    left, history = case["steps"], []
    while left > 0:
        n = min(left, case["every"])
        cav.step(n)
        left -= n
        ob = cav.observables()
        history.append([ob[k] for k in OBS])
    return dict(history=np.array(history), fields=cav.fields(out=state["out"]))


def work(case):
    """Bytes: the host arrays read and written, and the lattice (its
    populations, and the porosity where it varies) read once and written once
    per step, as in one pass over memory a step; operations: about 350 per
    node and step forward, three times that in the reverse sweep."""
    if case["kind"] == "sweep":
        nodes = sum(nx * ny for nx, ny in _sides(case))
        return dict(bytes=nodes * (152.0 * case["steps"] + 40), flops=350.0 * nodes * case["steps"])
    nodes = case["nx"] * case["ny"]
    field = case.get("porosity", "field") == "field"
    word = STORED[case["storage"]]
    step = 38.0 * word + (max(4, word) if field else 0)
    if case["kind"] == "adjoint":
        # forward, and a reverse step that reads the state and its adjoint and writes the adjoint
        return dict(bytes=nodes * (case["steps"] * (step + 57.0 * word) + 24 + word),
                    flops=4 * 350.0 * nodes * case["steps"])
    host = 8 * (5 + 2 + (1 if field else 0) + (3 if case["start"] == "fields" else 0))
    return dict(bytes=nodes * (case["steps"] * step + host), flops=350.0 * nodes * case["steps"])


# ---- the same in 64 bits -----------------------------------------------------

EX = (0, 1, 0, -1, 0, 1, -1, -1, 1)
EY = (0, 0, 1, 0, -1, 1, 1, -1, -1)
W9 = (4 / 9,) + (1 / 9,) * 4 + (1 / 36,) * 4
M9 = ((1, 1, 1, 1, 1, 1, 1, 1, 1), (-4, -1, -1, -1, -1, 2, 2, 2, 2), (4, -2, -2, -2, -2, 1, 1, 1, 1),
      (0, 1, 0, -1, 0, 1, -1, -1, 1), (0, -2, 0, 2, 0, 1, -1, -1, 1), (0, 0, 1, 0, -1, 1, 1, -1, -1),
      (0, 0, -2, 0, 2, 1, 1, -1, -1), (0, 1, -1, 1, -1, 0, 0, 0, 0), (0, 0, 0, 0, 0, 1, -1, 1, -1))
N5 = ((1, 1, 1, 1, 1), (0, 1, 0, -1, 0), (0, 0, 1, 0, -1), (-4, 1, 1, 1, 1), (0, 1, -1, 1, -1))
VARPI, S_E, S_EPS, S_Q, R_E, R_NU = 0.4, 1.1, 1.1, 1.2, 1.1, 1.1  # Sec. 4


def _root(s):
    """sqrt(s) with derivative 0 at s = 0."""
    pos = s > 0
    return torch.where(pos, torch.sqrt(torch.where(pos, s, torch.ones_like(s))), torch.zeros_like(s))


class _Exact:
    """The method on flat node lists; f is (9, n), gf and gs are (5, n)."""

    def __init__(self, nx, ny, kw, phi, H):
        dev, dt = phi.device, torch.float64
        self.nx, self.ny, self.phi = nx, ny, phi
        L = ny - 1.0
        uc = 0.1 / math.sqrt(3.0)
        nu = uc * L * math.sqrt(kw["Pr"] / kw["Ra"])
        alpha = nu / kw["Pr"]
        self.L, self.T0 = L, kw["T_ref"]
        self.gbeta = uc * uc / ((kw["T_hot"] - kw["T_cold"]) * L)
        self.sigma = kw["sigma"]
        self.local = bool(kw.get("hv_local", 0))
        self.hcoef = H * alpha / L**2
        Dp = 0.0135 * L
        self.hv_c = 0.376 * kw["Pr"]**0.37 * (Dp / nu)**0.644 * alpha / Dp**2
        if kw["permeability"] == LTNE_K_ERGUN:
            p = phi.detach()
            d = L * math.sqrt(150.0 * kw["Da"] / float((p**3 / (1 - p)**2).mean()))
            K = phi**3 * d * d / (150.0 * (1 - phi)**2)
        else:
            K = torch.full_like(phi, kw["Da"] * L * L)
        F = 1.75 / torch.sqrt(150.0 * phi**3) if kw["F_phi"] < 0 else kw["F_phi"]
        self.c0, self.c1 = nu / K, F / torch.sqrt(K)
        s_nu = 1 / (3 * nu + 0.5)
        za = 1 / (alpha * 2 / VARPI + 0.5)
        ea = 1 / (kw["gamma_sf"] / kw["sigma"] * alpha * 2 / VARPI + 0.5)
        col = lambda v: torch.tensor(v, dtype=dt, device=dev)[:, None]  # noqa: E731
        self.s = col([1, S_E, S_EPS, 1, S_Q, 1, S_Q, s_nu, s_nu])
        self.qf, self.qs = col([1, za, za, R_E, R_NU]), col([1, ea, ea, R_E, R_NU])
        self.M, self.N = (torch.tensor(a, dtype=dt, device=dev) for a in (M9, N5))
        self.Mi, self.Ni = torch.linalg.inv(self.M), torch.linalg.inv(self.N)
        self.w, self.ex, self.ey = col(W9), col(EX), col(EY)
        self.wt = col([1 - VARPI] + [VARPI / 4] * 4)
        # walls: node, the interior node it is rebuilt from, the imposed temperature
        node, near, temp = [], [], []
        for y in range(ny):
            for x in (range(nx) if y in (0, ny - 1) else (0, nx - 1)):
                node.append(y * nx + x)
                near.append(min(max(y, 1), ny - 2) * nx + min(max(x, 1), nx - 2))
                temp.append(kw["T_hot"] if x == 0 else kw["T_cold"] if x == nx - 1 else math.nan)
        self.node, self.near = (torch.tensor(v, device=dev) for v in (node, near))
        self.Tw = torch.tensor(temp, dtype=dt, device=dev)

    def macros(self, f, gf, gs, um, at=None):
        pick = (lambda v: v) if at is None else (lambda v: v[at])
        phi, c0, c1 = pick(self.phi), pick(self.c0), pick(self.c1)
        hv = self.hv_c * pick(um)**0.644 if self.local else self.hcoef
        a, b = hv / phi, hv / ((1 - phi) * self.sigma)
        Af, As = gf.sum(0), gs.sum(0)
        D = (Af - As) / (1 + a / 2 + b / 2)
        Sf, Ss = -a * D, b * D
        Tf, Ts = Af + Sf / 2, As + Ss / 2
        Gy = self.gbeta * (Tf - self.T0)
        rho = f.sum(0)
        vx = (self.ex * f).sum(0) / rho
        vy = (self.ey * f).sum(0) / rho + phi / 2 * Gy
        l0, l1 = (1 + phi / 2 * c0) / 2, phi / 2 * c1
        den = l0 + torch.sqrt(l0 * l0 + l1 * _root(vx * vx + vy * vy))
        ux, uy = vx / den, vy / den
        mag = _root(ux * ux + uy * uy)
        drag = c0 + c1 * mag
        return dict(rho=rho, ux=ux, uy=uy, Tf=Tf, Ts=Ts, Sf=Sf, Ss=Ss, mag=mag, phi=phi,
                    Fx=-phi * drag * ux, Fy=phi * (Gy - drag * uy))

    def equilibrium(self, m):
        eu = self.ex * m["ux"] + self.ey * m["uy"]
        u2 = (m["ux"]**2 + m["uy"]**2) / m["phi"]
        f = self.w * m["rho"] * (1 + 3 * eu + 4.5 * eu * eu / m["phi"] - 1.5 * u2)
        gf = self.wt * m["Tf"] + torch.where(self.wt == self.wt[0], 0.0, 0.5) * eu[:5] * m["Tf"] / m["phi"]
        return f, gf, self.wt * m["Ts"]

    def collide(self, f, gf, gs, m):
        rho, ux, uy, Fx, Fy, ip = m["rho"], m["ux"], m["uy"], m["Fx"], m["Fy"], 1 / m["phi"]
        u2, uF = 3 * rho * (ux * ux + uy * uy) * ip, 6 * rho * (ux * Fx + uy * Fy) * ip
        zero = torch.zeros_like(rho)
        meq = torch.stack([rho, -2 * rho + u2, rho - u2, rho * ux, -rho * ux, rho * uy, -rho * uy,
                           rho * (ux * ux - uy * uy) * ip, rho * ux * uy * ip])
        S = torch.stack([zero, uF, -uF, rho * Fx, -rho * Fx, rho * Fy, -rho * Fy,
                         2 * rho * (ux * Fx - uy * Fy) * ip, rho * (ux * Fy + uy * Fx) * ip])
        mm = self.M @ f
        f = self.Mi @ (mm - self.s * (mm - meq) + (1 - self.s / 2) * S)
        c3 = 5 * VARPI - 4
        out = []
        for g, q, T, Sr, adv in ((gf, self.qf, m["Tf"], m["Sf"], True), (gs, self.qs, m["Ts"], m["Ss"], False)):
            n = self.N @ g
            neq = torch.stack([T, ux * T * ip if adv else zero, uy * T * ip if adv else zero, c3 * T, zero])
            psi = torch.stack([Sr, zero, zero, c3 * Sr, zero])
            out.append(self.Ni @ (n - q * (n - neq) + (1 - q / 2) * psi))
        return f, out[0], out[1]

    def stream(self, p):
        v = p.view(-1, self.ny, self.nx)
        return torch.stack([torch.roll(v[i], (EY[i], EX[i]), (0, 1)) for i in range(len(v))]).view(len(v), -1)

    def step(self, f, gf, gs, m):
        """S_n and its macroscopic values to S_(n+1) and its."""
        um = m["mag"]
        f, gf, gs = (self.stream(p) for p in self.collide(f, gf, gs, m))
        near = self.near
        fr, gfr, gsr = f[:, near], gf[:, near], gs[:, near]
        r = self.macros(fr, gfr, gsr, um, near)
        fe, gfe, gse = self.equilibrium(r)
        free = torch.isnan(self.Tw)
        Tf, Ts = torch.where(free, r["Tf"], self.Tw), torch.where(free, r["Ts"], self.Tw)
        f = f.index_copy(1, self.node, self.w * r["rho"] + fr - fe)
        gf = gf.index_copy(1, self.node, self.wt * Tf + gfr - gfe)
        gs = gs.index_copy(1, self.node, self.wt * Ts + gsr - gse)
        return f, gf, gs, self.macros(f, gf, gs, um)

    def start(self, inputs):
        n = self.phi.numel()
        one = torch.ones(n, dtype=torch.float64, device=self.phi.device)
        take = lambda k, v: inputs[k].reshape(-1) if k in inputs else v * one  # noqa: E731
        m = dict(rho=take("rho", 1.0), ux=take("ux", 0.0), uy=take("uy", 0.0),
                 Tf=take("T_f", self.T0), Ts=take("T_s", self.T0), phi=self.phi)
        f, gf, gs = self.equilibrium(m)
        return f, gf, gs, self.macros(f, gf, gs, _root(m["ux"]**2 + m["uy"]**2))

    def nusselt(self, T, kw, hot):
        T = T.view(self.ny, self.nx)
        t1, t2 = (T[:, 1], T[:, 2]) if hot else (T[:, -2], T[:, -3])
        q = 1.5 * (kw["T_hot"] if hot else kw["T_cold"]) - 2 * t1 + 0.5 * t2
        q = q if hot else -q
        return (q.sum() - (q[0] + q[-1]) / 2) / (kw["T_hot"] - kw["T_cold"])

    def observables(self, m, kw):
        phi = self.phi
        energy = (phi * m["Tf"] + (1 - phi) * self.sigma * m["Ts"]).sum()
        vals = [self.nusselt(m["Tf"], kw, True), self.nusselt(m["Ts"], kw, True),
                self.nusselt(m["Tf"], kw, False), self.nusselt(m["Ts"], kw, False), m["rho"].sum(), energy,
                m["mag"].max(), (m["Tf"] - m["Ts"]).abs().max(), m["Tf"].mean(), m["Ts"].mean()]
        return [float(v) for v in vals]

    def fields(self, m):
        return {k: m[k].view(self.ny, self.nx).cpu().numpy() for k in FIELDS}


def _exact_cavity(nx, ny, kw, inputs, steps, every):
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    phi = inputs.get("porosity", torch.full((ny, nx), kw["porosity"], dtype=torch.float64, device=dev))
    with torch.no_grad():
        e = _Exact(nx, ny, kw, phi.reshape(-1), kw["H"])
        f, gf, gs, m = e.start(inputs)
        history = []
        for k in range(1, steps + 1):
            f, gf, gs, m = e.step(f, gf, gs, m)
            if k % every == 0 or k == steps:
                history.append(e.observables(m, kw))
        return np.array(history), e.fields(m)


def exact(case, seed):
    if case["kind"] == "sweep":
        got = [_exact_cavity(p["nx"], p["ny"], dict(p, F_phi=-1.0, permeability=LTNE_K_DARCY), {},
                             case["steps"], case["steps"]) for p in _sweep_params(case, seed)]
        return dict(observables=np.array([h[0] for h, _ in got]), fields=[f for _, f in got])
    kw, inputs = _keywords(case), _inputs(case, seed)
    if case["kind"] == "cavity":
        history, fields = _exact_cavity(case["nx"], case["ny"], kw, inputs, case["steps"], case["every"])
        return dict(history=history, fields=fields)
    from torch.utils.checkpoint import checkpoint

    phi = inputs.pop("porosity").reshape(-1).requires_grad_()
    H = torch.tensor(float(kw["H"]), dtype=torch.float64, device=phi.device, requires_grad=True)
    f, gf, gs, m = _Exact(case["nx"], case["ny"], kw, phi, H).start(inputs)

    def chunk(n, phi, H, f, gf, gs):
        e = _Exact(case["nx"], case["ny"], kw, phi, H)
        m = e.macros(f, gf, gs, None)
        for _ in range(n):
            f, gf, gs, m = e.step(f, gf, gs, m)
        return f, gf, gs

    left = case["steps"]
    while left > 0:
        n = min(left, 20)
        f, gf, gs = checkpoint(chunk, n, phi, H, f, gf, gs, use_reentrant=False)
        left -= n
    e = _Exact(case["nx"], case["ny"], kw, phi, H)
    m = e.macros(f, gf, gs, None)
    J = (e.nusselt(m["Tf"], kw, True) + e.nusselt(m["Ts"], kw, True)) / 2
    g_phi, g_H = torch.autograd.grad(J, (phi, H))
    return dict(J=float(J.detach()), dJ_dphi=g_phi.view(case["ny"], case["nx"]), dJ_dH=float(g_H))
