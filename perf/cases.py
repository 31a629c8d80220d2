"""The workloads whose speed this library answers for: what its users run, through its public
entry points (``LBE``, ``migration_loss``), over the sizes, storages and options in use.

A case is a dict of plain values:

``kind``     ``steps``: advance one handle by ``steps`` steps and read the fields of every instance;
             ``gradient``: the migration loss of ``steps`` steps and its gradients.
``problem``  the workload of ``paper_1412_6238_gb300.workloads`` the inputs come from.
``storage``  how the populations are held ("f64", "f32", "f16mix", "f16dev", "bf16dev").
``nx, ny``   cells (the sweep's instances have the sizes of ``batch_sweep``).
``rho2, interp, wall_mid, cos_wet, dissip``  options of ``lbe_params``, off when absent.

``exact`` is a plain torch FP64 statement of the scheme (Zheng, Zheng & Zhai, arXiv:1412.6238).
"""
import dataclasses
import math

import numpy as np
import torch

from paper_1412_6238_gb300 import workloads as wl
from paper_1412_6238_gb300.adjoint import MigrationProblem, migration_loss
from paper_1412_6238_gb300.lbe import LBE

OPTIONS = ("rho2", "interp", "wall_mid", "cos_wet", "dissip")
FIELDS = ("c", "p", "ux", "uy", "T")


def listed():
    return [
        # the two-layer thermal Poiseuille validation (FP64, 404 cells): a run
        # of many steps, each of which does next to nothing
        dict(name="channel_f64_4x101", kind="steps", problem="channel", nx=4, ny=101,
             storage="f64", steps=200),
        # the smoke check's drop: the smallest grid of the strip kernel
        dict(name="drop_f32_96x64", kind="steps", problem="drop", nx=96, ny=64, storage="f32",
             steps=200),
        # planar Marangoni convection, run for 100 000 steps in earnest, with
        # the steady-state check (residual and conserved sums) of such a run
        dict(name="planar_f32_512x256", kind="steps", problem="planar", nx=512, ny=256,
             storage="f32", steps=200, sums=True),
        # the migrating drop, run for 40 000 steps in earnest
        dict(name="drop_f32_512x1024", kind="steps", problem="drop", nx=512, ny=1024,
             storage="f32", steps=100),
        # the headline: the same drop scaled to 16.8 M cells (FP32), and to the
        # roofline sweep's other grid in the mixed storage
        dict(name="drop_f32_4096x4096", kind="steps", problem="drop", nx=4096, ny=4096,
             storage="f32", steps=20),
        dict(name="drop_f16mix_2048x4096", kind="steps", problem="drop", nx=2048, ny=4096,
             storage="f16mix", steps=20),
        # the smallest storage
        dict(name="drop_f16dev_2048x2048", kind="steps", problem="drop", nx=2048, ny=2048,
             storage="f16dev", steps=20),
        # the 64-drop parameter sweep of four grid sizes in one batch
        dict(name="sweep64_f16mix", kind="steps", problem="sweep", instances=64,
             storage="f16mix", steps=20),
        # a ragged grid, an odd number of steps, every boundary and property
        # variant on
        dict(name="wetting_f32_1000x777", kind="steps", problem="drop", nx=1000, ny=777,
             storage="f32", steps=51, interp=1, wall_mid=1, cos_wet=0.5),
        # a drop four times denser than its surroundings (FP64 only)
        dict(name="dense_f64_500x333", kind="steps", problem="drop", nx=500, ny=333,
             storage="f64", steps=20, rho2=4.0),
        # the dissipation term (FP32 on the tile kernel)
        dict(name="dissip_f32_512x256", kind="steps", problem="drop", nx=512, ny=256,
             storage="f32", steps=50, dissip=1),
        # the differentiable migration: loss and gradients (forward, reverse)
        dict(name="migration_f32_256x512", kind="gradient", problem="drop", nx=256, ny=512,
             storage="f32", steps=400, window=40, ckpt_every=100),
    ]


def _size(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """A case of the listed ones' ranges: any storage, any width and height
    (odd ones among them), each option where its storage has it."""
    what = rng.choice(["run", "run", "run", "run", "large", "batch", "option", "dense", "dissip",
                       "channel", "gradient"])
    if what == "channel":
        return dict(kind="steps", problem="channel", nx=rng.randint(4, 16),
                    ny=rng.randint(31, 301), storage="f64", steps=rng.randint(50, 200))
    if what == "batch":
        return dict(kind="steps", problem="sweep", instances=rng.randint(2, 24),
                    storage=rng.choice(["f16mix", "f32", "f16dev"]), steps=rng.randint(5, 20))
    if what == "gradient":
        n = rng.randint(60, 200)
        return dict(kind="gradient", problem="drop", nx=rng.randint(48, 256),
                    ny=rng.randint(64, 512), storage=rng.choice(["f32", "f32", "f16mix", "f64"]),
                    steps=n, window=rng.randint(1, n // 2), ckpt_every=rng.randint(20, 100))
    if what == "large":
        nx = rng.randint(1024, 4096)
        return dict(kind="steps", problem="drop", nx=nx, ny=rng.randint(1024, 4096),
                    storage=rng.choice(["f32", "f16mix", "f16dev", "bf16dev"]),
                    steps=rng.randint(5, 20))
    nx, ny = _size(rng, 40, 1200), _size(rng, 40, 1200)
    steps = max(10, min(200, int(2e7 / (nx * ny))))
    if what in ("dense", "dissip"):
        f64 = what == "dense" or rng.random() < 0.3
        c = dict(kind="steps", problem="drop", nx=nx, ny=ny, storage="f64" if f64 else "f32",
                 steps=max(4, min(50, int(2e6 / (nx * ny))) if f64 else steps))
        c["rho2" if what == "dense" else "dissip"] = rng.choice([0.25, 2.0, 4.0]) \
            if what == "dense" else 1
        return c
    if what == "option":
        return dict(kind="steps", problem="drop", nx=nx, ny=ny,
                    storage=rng.choice(["f32", "f16mix"]), steps=steps, interp=rng.randint(0, 1),
                    wall_mid=rng.randint(0, 1), cos_wet=round(rng.uniform(-0.8, 0.8), 3))
    c = dict(kind="steps", problem=rng.choice(["drop", "drop", "planar"]), nx=nx, ny=ny,
             storage=rng.choice(["f32", "f32", "f16mix", "f16dev", "bf16dev", "f64"]),
             steps=steps)
    if c["storage"] == "f64":
        c["steps"] = max(4, min(50, int(2e6 / (nx * ny))))
    if c["problem"] == "planar" and rng.random() < 0.5:
        c["sums"] = True
    return c


# ------------------------------------------------------------------ the inputs
def _workloads(case, seed):
    """The problem's workloads with a temperature perturbation of standard
    deviation 1e-4 drawn from the seed (as the migration problem has one)."""
    if case["problem"] == "channel":
        ws = [wl.layered_poiseuille(nx=case["nx"], ny=case["ny"])]
    elif case["problem"] == "planar":
        ws = [wl.planar_marangoni(nx=case["nx"], ny=case["ny"])]
    elif case["problem"] == "sweep":
        ws = wl.batch_sweep(case["instances"], seed=0)
    else:
        nx, ny = case["nx"], case["ny"]
        # radius min/8, in the middle or, with a contact angle, on the bottom
        # wall; small drops at the Reynolds number that keeps U = 6e-3
        R = max(5.0, min(nx, ny) / 8.0)
        yc = 0.8 * R if case.get("cos_wet") else ny / 2.0
        ws = [wl.droplet(nx, ny, R, nx / 2.0, yc, Re=min(1.0, R / 32.0), Ma=10.0, Ca=0.05,
                         eta_m=0.2, eta_r=0.5, lam_r=0.5)]
    rng = np.random.default_rng(seed)
    out = []
    for w in ws:
        p = dict(w.params)
        for k in OPTIONS:
            if k in case:
                p[k] = case[k]
        dT = rng.standard_normal(w.T0.shape, dtype=np.float32) * np.float32(1e-4)
        out.append(dataclasses.replace(w, params=p, T0=w.T0 + dT))
    return out


def _parameters(w):
    """sigmaT, eta2/eta1, lam2/lam1 of a workload."""
    p = w.params
    return p["sigmaT"], p["eta2"] / p["eta1"], p["lam2"] / p["lam1"]


def _perturbation(case, seed):
    rng = np.random.default_rng(seed + 1)
    return rng.standard_normal((case["ny"], case["nx"])) * 1e-4


def _dtype(case):
    return torch.float64 if case["storage"] == "f64" else torch.float32


def prepare(case, seed):
    ws = _workloads(case, seed)
    if case["kind"] == "gradient":
        dt = _dtype(case)
        leaf = [torch.tensor(v, dtype=dt, device="cuda", requires_grad=True)
                for v in _parameters(ws[0])]
        dT0 = torch.tensor(_perturbation(case, seed), dtype=dt, device="cuda", requires_grad=True)
        problem = MigrationProblem(ws[0], steps=case["steps"], window=case["window"],
                                   ckpt_every=case["ckpt_every"], storage=case["storage"])
        return dict(case=case, leaf=leaf + [dT0], problem=problem)
    sim = LBE(ws, storage=case["storage"])
    # the fields the program reads after its steps, in buffers it keeps
    bufs = [torch.empty((5,) + w.c0.shape, dtype=_dtype(case), device="cuda") for w in ws]
    outs = [{k: b[j] for j, k in enumerate(FIELDS)} for b in bufs]
    return dict(case=case, sim=sim, bufs=bufs, outs=outs)


def run(state):
    case = state["case"]
    if case["kind"] == "gradient":
        leaf = state["leaf"]
        loss = migration_loss(*leaf, state["problem"]).to(leaf[3].dtype)
        g = torch.autograd.grad(loss, leaf)
        return dict(loss=loss.detach(), sigmaT=g[0], eta_ratio=g[1], lam_ratio=g[2], dT0=g[3])
    sim = state["sim"]
    sim.step(case["steps"])
    for j, out in enumerate(state["outs"]):
        sim.fields(j, out=out)
    if case["problem"] == "sweep":
        return dict(fields=state["bufs"])
    res = dict(state["outs"][0])
    if case.get("sums"):
        s = sim.sums()
        res["sums"] = [s["sum_c"], s["sum_h"], s["residual"], s["nonfinite"]]
    return res


# bytes of a cell's 27 populations
STATE_BYTES = dict(f64=216, f32=108, f16mix=74, f16dev=56, bf16dev=56)


def work(case):
    """Per cell and step: the 27 populations read and written once, and about
    450 operations (moments 26, six stencils 120, normal and force 60, three
    collisions of nine directions 240).  A reverse step reads a stored state
    and an adjoint and writes an adjoint (27 FP64 values each) at about three
    times a step's operations, after one recomputed step.  The fields (and
    the state they come from) once per pass."""
    if case["problem"] == "sweep":
        cells = sum(w.cells for w in _sweep_shapes(case["instances"]))
    else:
        cells = case["nx"] * case["ny"]
    n, sb = case["steps"], STATE_BYTES[case["storage"]]
    fb = 8 if case["storage"] == "f64" else 4
    b, f = 2.0 * sb * n, 450.0 * n
    if case["kind"] == "gradient":
        b, f = 2 * b + 3 * 216.0 * n + 2 * fb, 2 * f + 1350.0 * n
    else:
        b, f = b + sb + 5 * fb, f + 250.0
    return dict(bytes=b * cells, flops=f * cells)


@dataclasses.dataclass
class _Shape:
    cells: int


def _sweep_shapes(n):
    """The grid sizes batch_sweep draws (seed 0), without building its fields."""
    rng = np.random.default_rng(0)
    out = []
    for _ in range(n):
        nx, ny = wl.BATCH_GRIDS[int(rng.integers(0, len(wl.BATCH_GRIDS)))]
        rng.uniform(size=5)
        out.append(_Shape(nx * ny))
    return out


# ------------------------------------------- the scheme in FP64, in plain torch
EX = (0, 1, 0, -1, 0, 1, -1, -1, 1)
EY = (0, 0, 1, 0, -1, 1, 1, -1, -1)
OPP = (0, 3, 4, 1, 2, 7, 8, 5, 6)
WT = (4 / 9,) + (1 / 9,) * 4 + (1 / 36,) * 4


class _Scheme:
    """One instance: state (27, ny, nx) of pre-collision populations."""

    def __init__(self, params, Tbot, Ttop, dev):
        self.P = dict(params)
        self.dev = dev
        t = lambda a: torch.as_tensor(np.asarray(a), dtype=torch.float64, device=dev)  # noqa: E731
        self.Tb, self.Tt = t(Tbot), t(Ttop)
        col = lambda v: t(v).reshape(9, 1, 1)  # noqa: E731
        self.ex, self.ey, self.w = col(EX), col(EY), col(WT)
        self.rho2 = self.P.get("rho2", 0.0) or self.P["rho"]
        self.vary = self.rho2 != self.P["rho"]

    def rho(self, c):
        return self.P["rho"] + c * (self.rho2 - self.P["rho"])

    def prop(self, a, b, c):
        if self.P.get("interp", 0):
            return 1 / ((1 - c) / a + c / b)
        return a + c * (b - a)

    # a field with `g` ghost rows on each side
    def ghost_c(self, c, g):
        kw = self.P.get("cos_wet", 0.0) * math.sqrt(2 * self.P["beta"]) / self.P["eps"]

        def row(j, m):
            return (m + (2 * j + 1) * kw * m * (1 - m))[None] if kw else m[None]

        lo = [row(j, c[j]) for j in reversed(range(g))]
        hi = [row(j, c[-1 - j]) for j in range(g)]
        return torch.cat(lo + [c] + hi)

    def ghost_T(self, T):
        return torch.cat([(2 * self.Tb - T[0])[None], T, (2 * self.Tt - T[-1])[None]])

    @staticmethod
    def ghost_p(p):
        return torch.cat([p[:1], p, p[-1:]])

    @staticmethod
    def ghost_u(u):
        return torch.cat([-u[:1], u, -u[-1:]])

    @staticmethod
    def at(e, i):
        """Neighbour i of every interior row of an extended field."""
        n = e.shape[0]
        r = e[1 + EY[i]:n - 1 + EY[i]]
        return torch.roll(r, -EX[i], 1) if EX[i] else r

    def grad(self, e):
        v = [self.at(e, i) for i in range(9)]
        gx = 3 * ((v[1] - v[3]) / 9 + ((v[5] - v[7]) + (v[8] - v[6])) / 36)
        gy = 3 * ((v[2] - v[4]) / 9 + ((v[5] - v[7]) - (v[8] - v[6])) / 36)
        return gx, gy

    def lap(self, e):
        v0 = e[1:-1]
        s = sum(WT[i] * (self.at(e, i) - v0) for i in range(1, 9))
        return 6 * s

    def drive(self, Q):
        """Moments, stencils, force, velocity and (varying density) p."""
        P = self.P
        f, c = Q[:9], Q[9:18].sum(0)
        rho = self.rho(c)
        T = Q[18:].sum(0) / (rho * P["cv"])
        p = f.sum(0)
        ce = self.ghost_c(c, 2)
        gx, gy = self.grad(ce)  # cells and one ghost row on each side
        inv = 1 / torch.sqrt(gx * gx + gy * gy + P["eta_n"] ** 2)
        kappa = self.grad(gx * inv)[0] + self.grad(gy * inv)[1]
        gcx, gcy = gx[1:-1], gy[1:-1]
        gTx, gTy = self.grad(self.ghost_T(T))
        mu = 2 * P["beta"] * c * (c - 1) * (2 * c - 1) - P["eps"] ** 2 * self.lap(ce[1:-1])
        sigma = P["sigma0"] - P["sigmaT"] * (T - P["Tref"])
        g2 = gcx * gcx + gcy * gcy
        pos = g2 > 0
        gabs = torch.where(pos, torch.sqrt(torch.where(pos, g2, torch.ones_like(g2))),
                           torch.zeros_like(g2))
        cdT = gcx * gTx + gcy * gTy
        ea = P["eps"] * 6 * math.sqrt(2.0)
        cap, mar = -sigma * kappa * ea * gabs, -P["sigmaT"] * ea
        Fx = cap * gcx + mar * (g2 * gTx - cdT * gcx) + rho * P["ax"]
        Fy = cap * gcy + mar * (g2 * gTy - cdT * gcy) + rho * P["ay"]
        jx = f[1] - f[3] + f[5] - f[6] - f[7] + f[8]
        jy = f[2] - f[4] + f[5] + f[6] - f[7] - f[8]
        ux, uy = 3 * jx / rho + Fx / (2 * rho), 3 * jy / rho + Fy / (2 * rho)
        dR = None
        if self.vary:
            dR = ((self.rho2 - P["rho"]) / 3 * gcx, (self.rho2 - P["rho"]) / 3 * gcy)
            p = p + 0.5 * (ux * dR[0] + uy * dR[1])
        return c, p, T, rho, mu, Fx, Fy, ux, uy, dR

    def fields(self, Q):
        c, p, T, _, _, _, _, ux, uy, _ = self.drive(Q)
        return dict(c=c, p=p, ux=ux, uy=uy, T=T)

    def step(self, Q):
        P, w, ex, ey = self.P, self.w, self.ex, self.ey
        c, p, T, rho, mu, Fx, Fy, ux, uy, dR = self.drive(Q)
        gpx, gpy = self.grad(self.ghost_p(p))
        f, g, h = Q[:9], Q[9:18], Q[18:]
        rcs = rho / 3
        om_f = 1 / (self.prop(P["eta1"], P["eta2"], c) / rcs + 0.5)
        om_T = 2 / (2 * self.prop(P["lam1"], P["lam2"], c) / (rcs * P["cv"]) + 1)
        om_g = 1 / P["tau_g"]
        Gm = P["mobility"] / (P["tau_g"] - 0.5)
        xu = 3 * (ex * ux + ey * uy)
        q = xu + 0.5 * (xu * xu - 3 * (ux * ux + uy * uy))
        G = w * (1 + q)
        dx, dy = ex - ux, ey - uy
        src = (Fx * dx + Fy * dy) * G
        Bx, By = Fx - gpx, Fy - gpy
        if dR is not None:
            src = src + (dx * dR[0] + dy * dR[1]) * (G - w)
        fo = f - om_f * (f - w * (p + rcs * q)) + (1 - 0.5 * om_f) * src
        H = (3 * Gm * mu).expand(9, -1, -1)
        H = torch.cat([((c - (1 - WT[0]) * 3 * Gm * mu) / WT[0])[None], H[1:]])
        go = g - om_g * (g - w * (H + c * q)) + \
            (1 - 0.5 * om_g) * (c * (dx * Bx + dy * By) / rcs * G)
        heq = rho * P["cv"] * T * G
        if dR is not None:
            Bx, By = Bx + dR[0], By + dR[1]
        hs = (Bx * dx + By * dy) / rcs * heq
        aT = 1 - 0.5 * om_T
        ho = h - om_T * (h - heq) + aT * hs
        if P.get("dissip", 0):
            a, b = self.grad(self.ghost_u(ux))
            d, e = self.grad(self.ghost_u(uy))
            fbe = rho * G
            fph = fbe + (1 - 0.5 * om_f) * (3 * (f - w * (p - rcs)) - fbe)
            S = -fph * (dx * (ex * a + ey * b) + dy * (ex * d + ey * e))
            S0 = S.sum(0)
            ho = ho + aT * (S - w * S0) + w * S0
        return self.stream(torch.cat([fo, go, ho]))

    def stream(self, post):
        out = [None] * 27
        for k in (0, 1, 2):
            for i in range(9):
                v = post[9 * k + i]
                v = torch.roll(v, EX[i], 1) if EX[i] else v
                if EY[i]:
                    wrow = 0 if EY[i] > 0 else -1
                    back = post[9 * k + OPP[i]][wrow]
                    if k == 2:
                        Tw = self.Tb if EY[i] > 0 else self.Tt
                        if self.P.get("wall_mid", 0) and EX[i]:
                            Tw = 0.5 * (Tw + torch.roll(Tw, EX[i]))
                        cn = sum(out[9 + j][wrow] for j in range(9))
                        back = -back + 2 * WT[i] * self.rho(cn) * self.P["cv"] * Tw
                    v = torch.cat([back[None], v[:-1]] if EY[i] > 0 else [v[1:], back[None]])
                out[9 * k + i] = v
        return torch.stack(out)

    def rest(self, c0, T0):
        P = self.P
        mu = 2 * P["beta"] * c0 * (c0 - 1) * (2 * c0 - 1) - \
            P["eps"] ** 2 * self.lap(self.ghost_c(c0, 1))
        Gm = 3 * P["mobility"] / (P["tau_g"] - 0.5)
        g0 = c0 - (1 - WT[0]) * Gm * mu
        g = [g0] + [WT[i] * Gm * mu for i in range(1, 9)]
        h = [WT[i] * self.rho(c0) * P["cv"] * T0 for i in range(9)]
        return torch.stack([torch.zeros_like(c0)] * 9 + g + h)


def exact(case, seed):
    dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")
    ws = _workloads(case, seed)
    if case["kind"] == "gradient":
        return _exact_gradient(case, seed, ws[0], dev)
    if case["problem"] == "planar" and case["ny"] * case["nx"] * case["steps"] > 1e9:
        return None
    out = []
    with torch.no_grad():
        for w in ws:
            S = _Scheme(w.params, w.Tbot, w.Ttop, dev)
            Q = S.rest(torch.as_tensor(w.c0, device=dev), torch.as_tensor(w.T0, device=dev))
            prev = None
            for n in range(case["steps"]):
                prev = Q if n == case["steps"] - 1 else None
                Q = S.step(Q)
            F = S.fields(Q)
            if case.get("sums"):
                A = S.fields(prev)
                du = sum(((F[k] - A[k]) ** 2).sum() for k in ("ux", "uy"))
                uu = sum((F[k] ** 2).sum() for k in ("ux", "uy"))
                F["sums"] = [float(F["c"].sum()), float(Q[18:].sum()), float((du / uu).sqrt()), 0]
            out.append(F)
    if case["problem"] == "sweep":
        return dict(fields=[torch.stack([F[k] for k in FIELDS]) for F in out])
    if case["problem"] == "channel":  # p and u_y are zero but for rounding
        out[0]["p"] = out[0]["uy"] = None
    return out[0]


def _exact_gradient(case, seed, w, dev):
    """Autograd through the FP64 scheme, in segments recomputed from their
    first state."""
    n, win = case["steps"], case["window"]
    dt = _dtype(case)
    # the values the program holds (of its own type)
    v = [float(torch.tensor(x, dtype=dt)) for x in _parameters(w)]
    dT0 = torch.tensor(_perturbation(case, seed), dtype=dt).to(dev, torch.float64)
    leaf = [torch.tensor(x, dtype=torch.float64, device=dev, requires_grad=True) for x in v]
    T0 = torch.as_tensor(w.T0, device=dev) + dT0

    def scheme():
        p = dict(w.params)
        p["sigmaT"], p["eta2"], p["lam2"] = leaf[0], leaf[1] * p["eta1"], leaf[2] * p["lam1"]
        return _Scheme(p, w.Tbot, w.Ttop, dev)

    def observable(S, Q):
        F = S.fields(Q)
        return (F["c"] * F["uy"]).sum() / F["c"].sum()

    def span(Q, a, b):
        """States a..b from state a, and the loss of states a+1..b."""
        S, L = scheme(), torch.zeros((), dtype=torch.float64, device=dev)
        for j in range(a + 1, b + 1):
            Q = S.step(Q)
            if j > n - win:
                L = L + observable(S, Q) / win
        return Q, L

    K = 20
    with torch.no_grad():
        Q = scheme().rest(torch.as_tensor(w.c0, device=dev), T0)
        keep, loss = [], 0.0
        for a in range(0, n, K):
            keep.append(Q)
            Q, L = span(Q, a, min(n, a + K))
            loss = loss + L
    adj = torch.zeros_like(Q)
    grads = [torch.zeros_like(x) for x in leaf]
    for a in reversed(range(0, n, K)):
        Q = keep.pop().requires_grad_(True)
        Qb, L = span(Q, a, min(n, a + K))
        # (the loss part is a constant in segments before the window)
        tot = (Qb * adj).sum() + L
        got = torch.autograd.grad(tot, [Q] + leaf)
        adj = got[0]
        grads = [x + y for x, y in zip(grads, got[1:])]
    P = w.params
    wts = torch.tensor(WT, dtype=torch.float64, device=dev).reshape(9, 1, 1)
    return dict(loss=loss, sigmaT=grads[0], eta_ratio=grads[1], lam_ratio=grads[2],
                dT0=P["rho"] * P["cv"] * (wts * adj[18:]).sum(0))
