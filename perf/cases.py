"""Timed cases of the solver: what programs that use it call, over the sizes they use.

A case is a dict of plain values.  Its "kind" says which calls one pass makes:

  steps   a state goes in, `steps` implicit time steps run, the new state comes
          out (the loop of a simulation, and a served request's share of it);
          "host" moves the fields as numpy arrays, else as CUDA tensors
  vcycle  one outer cycle of a step by hand: qnsch_begin_step, qnsch_vcycle,
          qnsch_commit_step (convergence studies, tuning of the smoother)
  batch   the same for several instances advanced together (qnsch_batch_step)
  record  what a simulation logs of a state: mass, energy, the diagnostics of
          the experiments and the divergence field
  mass    the allocation-free mass reduction on a caller's tensor

Inputs are the diffuse-interface scenes of the paper's experiments with their
geometry drawn from the seed, plus a smooth flow, so that every term acts.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1703_06606_gb300 import qnsch

FIELDS = ("c", "mu", "u", "v", "p")

# Solver options by path: the smoothing counts, predictor and launch thresholds
# that the repository's benchmark and its server run with.
PATHS = {
    "fp64": dict(nu1=1, nu2=1, nu1_fine=2, nu2_fine=3, predictor=2),
    "fp64_default": dict(),
    "mixed": dict(precision=1, nu1=1, nu2=1, nu1_fine=2, nu2_fine=3, predictor=2),
    "mixed_12": dict(precision=1, nu1=1, nu2=2, predictor=2),
    "fp64_coupled": dict(coupled=1, nu1=1, nu2=2, predictor=2),
    "mixed_coupled": dict(precision=1, coupled=1, nu1=1, nu2=2, predictor=2),
    "served": dict(precision=1, coupled=1, fuse_cells32=2048, vanka_team_max32=0, nu1=1, nu2=2,
                   predictor=2),
    "projection": dict(scheme=1, nu1=1, nu2=2, predictor=2),
}


def listed():
    return [
        # A small wave on the host path, as the run command drives it: the
        # shortest simulation there is, where launches and latency count.
        dict(name="capillary_64x64_fp64_host", kind="steps", scene="capillary", m1=64, m2=64,
             periodic=True, path="fp64", steps=1, dt=1e-3, ratio=1.0, eta_ratio=1.0, host=True),
        # The benchmark's headline: the rising droplet in FP64 with the paper's
        # smoother; three steps, so that a step that follows a step is in it.
        dict(name="drop_256x512_fp64", kind="steps", scene="drop", m1=256, m2=512, periodic=False,
             path="fp64", steps=3, dt=2e-4, ratio=10.0, eta_ratio=10.0, host=False),
        # The same droplet by FP32 cycles under the FP64 defect correction.
        dict(name="drop_256x512_mixed", kind="steps", scene="drop", m1=256, m2=512,
             periodic=False, path="mixed", steps=3, dt=2e-4, ratio=10.0, eta_ratio=10.0,
             host=False),
        # The largest instance of the droplet batch, alone, with the coupled block.
        dict(name="drop_512x512_mixed_coupled", kind="steps", scene="drop", m1=512, m2=512,
             periodic=False, path="mixed_coupled", steps=1, dt=2e-4, ratio=50.0, eta_ratio=20.0,
             host=False),
        # Rayleigh-Taylor at its full size: the largest grid a single run uses.
        dict(name="rayleigh_taylor_1024x4096_mixed", kind="steps", scene="rt", m1=1024, m2=4096,
             periodic=True, path="mixed_12", steps=1, dt=1e-4, ratio=3.0, eta_ratio=1.0,
             host=False),
        # A served request of a middling odd size (448 = 7 x 64) with the
        # server's options.
        dict(name="capillary_448x448_served", kind="steps", scene="capillary", m1=448, m2=448,
             periodic=True, path="served", steps=2, dt=1e-4, ratio=1.0, eta_ratio=1.0,
             host=False),
        # The paper's projection method, as its cost table compares the methods.
        dict(name="drop_128x256_projection", kind="steps", scene="drop", m1=128, m2=256,
             periodic=True, path="projection", steps=1, dt=2e-4, ratio=10.0, eta_ratio=10.0,
             host=False),
        # A ragged grid (it coarsens to 6 x 9) with the coupled block in FP64.
        dict(name="drop_96x144_fp64_coupled", kind="steps", scene="drop", m1=96, m2=144,
             periodic=False, path="fp64_coupled", steps=1, dt=4e-4, ratio=10.0, eta_ratio=5.0,
             host=False),
        # One outer cycle with the library's default counts on a periodic grid.
        dict(name="vcycle_256x256_fp64", kind="vcycle", scene="capillary", m1=256, m2=256,
             periodic=True, path="fp64_default", dt=2e-4, ratio=3.0, eta_ratio=2.0),
        # A batch of droplets of mixed sizes in flight at once.
        dict(name="batch_12_drops", kind="batch", count=12, scene="drop", small=64, large=256,
             periodic=False, path="served", dt=2e-4, ratio=20.0, eta_ratio=10.0),
        # What a simulation logs after a step.
        dict(name="record_256x512", kind="record", scene="drop", m1=256, m2=512, periodic=False,
             path="fp64_default", ratio=10.0, eta_ratio=10.0),
        # The mass of a caller's field, at the largest size the call takes.
        dict(name="mass_2048x4096", kind="mass", scene="rt", m1=2048, m2=4096, periodic=True,
             ratio=3.0),
    ]


def draw(rng):
    kind = rng.choice(["steps"] * 7 + ["vcycle", "record", "mass", "batch"])
    periodic = rng.random() < 0.5
    ratio = round(10.0 ** rng.uniform(0.0, 2.0), 3)
    eta_ratio = round(10.0 ** rng.uniform(0.0, 1.3), 3)
    if kind == "mass":  # any size up to the call's limit, odd ones among them
        m1 = int(2 ** rng.uniform(5.0, 11.5))
        return dict(kind=kind, scene="rt", m1=m1, m2=int(m1 * rng.uniform(0.5, 2.0)),
                    periodic=periodic, ratio=ratio)
    scene = rng.choice(["drop", "capillary"])
    if kind == "batch":
        return dict(kind=kind, count=rng.randint(2, 10), scene="drop",
                    small=rng.choice([48, 64, 80]), large=rng.choice([96, 128, 192, 256]),
                    periodic=False, path="served", dt=2e-4, ratio=ratio, eta_ratio=eta_ratio)
    # sides q 2^n: they coarsen to q cells, as the served sizes (multiples of 64) do
    q, top = rng.choice([4, 5, 6, 7]), rng.uniform(5.0, 9.1)
    m1 = q << max(3, int(top - math.log2(q) + 0.5))
    m2 = rng.choice([m1, m1, m1 * 3 // 2, 2 * m1])
    if kind == "record":  # no multigrid work: any size
        m1, m2 = m1 + rng.randint(0, 9) * 2, m2 + rng.randint(0, 19)
    h = 1.0 / m1
    case = dict(kind=kind, scene=scene, m1=m1, m2=m2, periodic=periodic,
                path="fp64_default", ratio=ratio, eta_ratio=eta_ratio)
    if kind == "record":
        return case
    case["dt"] = round(rng.uniform(0.03, 0.08) * min(h, 1.0 / 64), 7)
    if kind == "steps":
        case.update(path=rng.choice(["fp64", "mixed", "fp64_coupled", "mixed_coupled", "served",
                                     "fp64_default"] + (["projection"] if m1 <= 256 else [])),
                    steps=rng.randint(1, 2), host=rng.random() < 0.25)
    if "coupled" not in PATHS[case["path"]]:
        # the paper's separate smoothers stall at high ratios: the coupled block is for those
        case["ratio"] = round(ratio ** 0.45, 3)
    return case


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def physics(case, m1):
    """Creation parameters of an instance (the experiments' numbers).  c = 1 is
    the drop or the lower fluid: heavier by `ratio` and more viscous by
    `eta_ratio` under a capillary wave, lighter and less viscous else."""
    rt = case["scene"] == "rt"
    up = 1.0 if case["scene"] == "capillary" else -1.0
    Cn = 0.005 if rt else max(0.01, 2.5 / m1)
    return dict(Lx=1.0, periodic_x=case["periodic"], rho1=case["ratio"] ** up, rho2=1.0,
                eta1=case.get("eta_ratio", 1.0) ** up, eta2=1.0, Re=3000.0 if rt else 35.0,
                We=200.0 if rt else 10.0, Pe=1.0 / Cn, Cn=Cn, Fr=1.0)


def scene(case, m1, m2, seed):
    """The fields of a state, FP64 CUDA tensors in the library's layouts."""
    rng = np.random.default_rng(seed)
    dev = torch.device("cuda")
    h, Ly = 1.0 / m1, m2 / m1
    x = (torch.arange(m1, device=dev, dtype=torch.float64) + 0.5) * h
    y = (torch.arange(m2, device=dev, dtype=torch.float64)[:, None] + 0.5) * h
    Cn = physics(case, m1)["Cn"]
    if case["scene"] == "drop":
        R, x0 = rng.uniform(0.2, 0.28), 0.5 + rng.uniform(-0.05, 0.05)
        d = torch.sqrt((x - x0) ** 2 + (y - min(0.5, 0.5 * Ly) * rng.uniform(0.95, 1.05)) ** 2) - R
    else:
        amp = rng.uniform(0.08, 0.12) if case["scene"] == "rt" else rng.uniform(0.01, 0.03)
        d = y - 0.5 * Ly * rng.uniform(0.95, 1.05) - amp * torch.cos(2.0 * math.pi * x)
    c = 0.5 * (1.0 - torch.tanh(d / (2.0 * math.sqrt(2.0) * Cn)))
    # a flow from a stream function at the vertices, zero on the walls, and a
    # weak compressible part, as a step of fluids of unequal density leaves one
    xe = torch.arange(m1 + 1, device=dev, dtype=torch.float64) * h
    ye = torch.arange(m2 + 1, device=dev, dtype=torch.float64)[:, None] * h
    phase = rng.uniform(0.0, 2.0 * math.pi)
    wx = torch.sin(2.0 * math.pi * xe + phase) if case["periodic"] else torch.sin(math.pi * xe) ** 2
    psi = rng.uniform(0.005, 0.015) * wx * torch.sin(math.pi * ye / Ly) ** 2
    u = (psi[1:] - psi[:-1]) / h + 1e-3 * torch.sin(math.pi * y / Ly) * torch.sin(2.0 * math.pi * xe)
    v = -(psi[:, 1:] - psi[:, :-1]) / h
    v = v + 1e-3 * torch.sin(math.pi * ye / Ly) * torch.cos(2.0 * math.pi * x)
    if not case["periodic"]:
        u[:, 0] = u[:, -1] = 0.0
    else:
        u[:, 0] = u[:, -1]
    v[0] = v[-1] = 0.0
    z = torch.zeros_like(c)
    return {"c": c.contiguous(), "mu": z, "p": z.clone(), "u": u.contiguous(), "v": v.contiguous()}


def sizes(case, seed):
    """Grids of a batch: small, middling and large ones in turn."""
    return [(m, m) for k in range(case["count"])
            for m in [(case["small"], case["large"], 2 * case["small"])[k % 3]]]


def prepare(case, seed):
    st = {"case": case}
    if case["kind"] == "mass":
        st["c"] = scene(case, case["m1"], case["m2"], seed)["c"]
        st["out"] = torch.zeros(2, dtype=torch.float64, device="cuda")
        return st
    grids = sizes(case, seed) if case["kind"] == "batch" else [(case["m1"], case["m2"])]
    st["solvers"], st["in"], st["out"] = [], [], []
    for n, (m1, m2) in enumerate(grids):
        s = qnsch.Solver(m1, m2, tol=1e-9, **physics(case, m1), **PATHS[case["path"]])
        f = scene(case, m1, m2, seed * 1000 + n)
        if case.get("host"):
            f = {k: t.cpu().numpy() for k, t in f.items()}
        else:
            st["out"].append({k: torch.empty_like(t) for k, t in f.items()})
        st["solvers"].append(s)
        st["in"].append(f)
    if case["kind"] == "batch":
        st["batch"] = qnsch.Batch(st["solvers"])
    if case["kind"] == "record":
        st["solvers"][0].set_fields_device(st["in"][0])
    torch.cuda.synchronize()
    return st


def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "mass":
        q = physics(case, case["m1"])
        qnsch.mass_noalloc(st["c"], 1.0 / case["m1"], q["rho1"], q["rho2"], st["out"])
        return st["out"]
    s = st["solvers"][0]
    if kind == "record":
        m, e = s.mass(), s.energy()
        return {"mass": list(m), "energy": e[0], "diagnostics": s.diagnostics(),
                "divergence": s.divergence()}
    if case.get("host"):
        s.set_fields(st["in"][0])
        for _ in range(case["steps"]):
            s.step(case["dt"])
        return s.get_fields()
    for s, f in zip(st["solvers"], st["in"]):
        s.set_fields_device(f)
    if kind == "batch":
        status, _ = st["batch"].step(case["dt"])
        if any(status):
            raise RuntimeError("a member's step failed: %s" % status)
    elif kind == "vcycle":
        s.begin_step(case["dt"])
        s.vcycle()
        s.commit_step()
    else:
        for _ in range(case["steps"]):
            s.step(case["dt"])
    for s, o in zip(st["solvers"], st["out"]):
        s.get_fields_device(o)
    return st["out"]


# ---------------------------------------------------------------------------
# work
# ---------------------------------------------------------------------------
def work(case):
    """Bytes: the state in and out (the field for the reductions).  Operations:
    of a step, four outer cycles (a predicted start needs as many at least) of
    the path's smoothing steps on every level, at 450 operations a cell and
    smoothing step (a 2x2 Newton step, a 5x5 block solve and their residuals)."""
    if case["kind"] == "mass":
        n = case["m1"] * case["m2"]
        return {"bytes": 8.0 * n + 16.0, "flops": 6.0 * n}
    cells = sum(a * b for a, b in (sizes(case, 0) if case["kind"] == "batch"
                                   else [(case["m1"], case["m2"])]))
    if case["kind"] == "record":
        return {"bytes": 8.0 * 4.0 * cells, "flops": 80.0 * cells}
    o = PATHS[case["path"]]
    nu1, nu2 = o.get("nu1", 2), o.get("nu2", 2)
    fine = o.get("nu1_fine", nu1) + o.get("nu2_fine", nu2)
    per_cycle = 450.0 * (fine + (nu1 + nu2) / 3.0)
    cycles = 1 if case["kind"] == "vcycle" else 4 * case.get("steps", 1)
    return {"bytes": 80.0 * cells, "flops": per_cycle * cycles * cells}


# ---------------------------------------------------------------------------
# the same outputs in 64 bits from the discrete equations, in torch
# ---------------------------------------------------------------------------
def _gap(r1, r2):
    """eta(rho1, rho2), the surface-tension ratio; a series near rho1 = rho2."""
    q = r2 / r1 - 1.0
    if abs(q) < 0.1:
        s = sum(2.0 * (-1.0) ** n * q ** n / ((n + 2.0) * (n + 3.0)) for n in range(24))
        return 1.0 / (2.0 * math.sqrt(2.0) * r1 * (1.0 + q) * s)
    return (r2 - r1) ** 3 / (2.0 * math.sqrt(2.0) * r1 * r2 *
                             (r2 * r2 - r1 * r1 - 2.0 * r1 * r2 * math.log(r2 / r1)))


class _Grid:
    """Neighbour values on the staggered grid.  Every unknown is a (m2, m1)
    array: u at the cell's east edge, v at its north edge (zero on a wall)."""

    def __init__(self, px):
        self.px = px

    def _x(self, a, n, edge):
        b = torch.roll(a, -n, 1)
        if not self.px:
            at = -1 if n == 1 else 0
            col = torch.zeros_like(b)
            col[:, at] = 1.0
            b = torch.where(col > 0, edge, b)
        return b

    def _y(self, a, n, edge):
        b = torch.roll(a, -n, 0)
        row = torch.zeros_like(b)
        row[-1 if n == 1 else 0] = 1.0
        return torch.where(row > 0, edge, b)

    def cell(self, a):  # east, west, north, south neighbours of a cell value
        return self._x(a, 1, a), self._x(a, -1, a), self._y(a, 1, a), self._y(a, -1, a)

    def E(self, a):
        return self._x(a, 1, a)

    def N(self, a):
        return self._y(a, 1, a)

    def u(self, a):
        o = torch.zeros_like(a)
        return self._x(a, 1, o), self._x(a, -1, o), self._y(a, 1, -a), self._y(a, -1, -a)

    def v(self, a):
        o = torch.zeros_like(a)
        return self._x(a, 1, -a), self._x(a, -1, -a), self._y(a, 1, o), self._y(a, -1, o)


class _Step:
    """The fully discrete scheme of one step (the primitive method, or the
    projection method) from the state (c, mu, u, v, p) as its residual."""

    def __init__(self, q, dt, state, projection):
        self.q, self.idt, self.projection = q, 1.0 / dt, projection
        self.G = G = _Grid(q["periodic_x"])
        r1, r2 = q["rho1"], q["rho2"]
        self.al = (r2 - r1) / (r1 * r2)
        self.vis = lambda c: 1.0 / ((q["eta2"] - q["eta1"]) / (q["eta1"] * q["eta2"]) * c +
                                    1.0 / q["eta2"])
        self.rho = lambda c: 1.0 / (self.al * c + 1.0 / r2)
        M = q["Cn"]
        self.M, eta = M, _gap(r1, r2)
        self.K, self.Lam = M * eta / (q["Cn"] * q["We"]), q["Cn"] * eta * M / q["We"]
        self.Fri = 1.0 / q["Fr"]
        c, _, u, v, _ = state
        m2, m1 = c.shape
        self.h = h = q["Lx"] / m1
        self.wu = torch.ones_like(c)  # 1 on the edges that hold an unknown
        self.wv = torch.ones_like(c)
        self.wv[-1] = 0.0
        if not q["periodic_x"]:
            self.wu[:, -1] = 0.0
        self.c, self.u, self.v = c, u, v
        self.rn, self.mn, self.vn_ = self.rho(c), torch.sqrt((c * (1 - c)) ** 2 + q["Cn"]), self.vis(c)
        self.Gn = self.grad2(c)
        uE, uW, uN, _ = G.u(u)
        vE, _, vN, vS = G.v(v)
        rE, _, rN, _ = G.cell(self.rn)
        self.Ax, self.Ay = 0.5 * (self.rn + rE), 0.5 * (self.rn + rN)
        self.Sx, self.Sy = self.rn * 0.5 * (u + uW), self.rn * 0.5 * (v + vS)
        corner = 0.25 * (self.rn + rE + rN + G.E(rN))  # at (i + 1/2, j + 1/2)
        self.Qx, self.Qy = corner * 0.5 * (vE + v), corner * 0.5 * (uN + u)
        self.muv = 0.25 * (self.vn_ + G.E(self.vn_) + G.N(self.vn_) + G.E(G.N(self.vn_)))
        # the vertices below and to the left: on a wall the edges' mean velocity
        # is zero and the viscosity that of the wall's two cells
        z = torch.zeros_like(c)
        self.QxS, self.QyW = G._y(self.Qx, -1, z), G._x(self.Qy, -1, z)
        self.muvS = G._y(self.muv, -1, 0.5 * (self.vn_ + G.E(self.vn_)))
        self.muvW = G._x(self.muv, -1, 0.5 * (self.vn_ + G.N(self.vn_)))
        self.Dcx, self.Dcy = (G.E(c) - c) / h, (G.N(c) - c) / h

    def grad2(self, c):
        e, w, n, s = self.G.cell(c)
        return 0.5 * ((e - c) ** 2 + (c - w) ** 2 + (n - c) ** 2 + (c - s) ** 2) / self.h ** 2

    def div(self, k, f):  # div of (A k) grad f
        G = self.G
        return sum(0.5 * (a + k) * (b - f) for a, b in zip(G.cell(k), G.cell(f))) / self.h ** 2

    def velocity(self, c, mu, u, v, p):
        """u^{n+1}, v^{n+1}: the iterate's own, or those of the projection equation."""
        if not self.projection:
            return u, v
        G, h, r = self.G, self.h, self.rho(c)

        def face(f, x, g):
            st = 0.5 * (f(r) * mu + r * f(mu)) * (f(c) - c) / h - (f(p) - p) / h
            return x + st / (self.M * 0.5 * (r + f(r)) * self.idt) - g / self.idt
        return face(G.E, u, 0.0) * self.wu, face(G.N, v, self.Fri) * self.wv

    def residual(self, X):
        q, G, h, idt = self.q, self.G, self.h, self.idt
        c, mu, u, v, p = X
        cn, rn, mn, al = self.c, self.rn, self.mn, self.al
        r = self.rho(c)
        flux = self.div(mn, mu) + al * self.div(mn, p)
        uu, vv = self.velocity(c, mu, u, v, p)
        _, uW, _, _ = G.u(uu)
        _, _, _, vS = G.v(vv)
        ra, ca = (r, c) if self.projection else (rn, cn)
        rE, rW, rN, rS = G.cell(ra)
        cE, cW, cN, cS = G.cell(ca)
        adv = 0.5 / h * (rE * (cE - ca) * uu + rW * (ca - cW) * uW + rN * (cN - ca) * vv +
                         rS * (ca - cS) * vS)
        r0 = rn if self.projection else r
        Rc = r0 * (c - cn) * idt + adv - flux / q["Pe"]
        Rp = (uu - uW + vv - vS) / h - al * flux / q["Pe"]
        rh, sec = 0.5 * (r + rn), -al * r * rn
        F = lambda a: 0.25 * (a * (a - 1.0)) ** 2  # noqa: E731
        g = 0.25 * (c * (c - 1.0) + cn * (cn - 1.0)) * (c + cn - 1.0)
        Rm = (r0 * mu - self.K * (rh * g + 0.5 * (F(c) + F(cn)) * sec) -
              0.25 * self.Lam * (self.grad2(c) + self.Gn) * sec + self.Lam * self.div(rh, 0.5 * (c + cn)))
        # momentum rows at the east and north edges
        uE, uW, uN, uS = G.u(u)
        vE, vW, vN, vS = G.v(v)
        dx, dxE = (u - uW) / h, (uE - u) / h
        d, dE = dx + (v - vS) / h, dxE + (vE - G._y(vE, -1, torch.zeros_like(v))) / h
        top, bot = (uN - u) / h, (u - uS) / h
        Ru = (self.Ax * (u - self.u) * idt +
              0.5 * (G.E(self.Sx) * dxE + self.Sx * dx + self.Qx * top + self.QxS * bot) +
              0.5 * (0.5 * (r + G.E(r)) - self.Ax) * idt * u +
              0.5 * ((G.E(self.Sx) - self.Sx) + (self.Qx - self.QxS)) / h * u -
              ((G.E(self.vn_) * dxE - self.vn_ * dx) + (self.muv * top - self.muvS * bot) +
               (G.E(self.vn_) * dE - self.vn_ * d) / 3.0) / (h * q["Re"]))
        dy, dyN = (v - vS) / h, (vN - v) / h
        uNW = G._x(uN, -1, torch.zeros_like(u))
        d, dN = dy + (u - uW) / h, dyN + (uN - uNW) / h
        rgt, lft = (vE - v) / h, (v - vW) / h
        Rv = (self.Ay * (v - self.v) * idt +
              0.5 * (self.Qy * rgt + self.QyW * lft + G.N(self.Sy) * dyN + self.Sy * dy) +
              0.5 * (0.5 * (r + G.N(r)) - self.Ay) * idt * v +
              0.5 * ((self.Qy - self.QyW) + (G.N(self.Sy) - self.Sy)) / h * v -
              ((self.muv * rgt - self.muvW * lft) + (G.N(self.vn_) * dyN - self.vn_ * dy) +
               (G.N(self.vn_) * dN - self.vn_ * d) / 3.0) / (h * q["Re"]))
        if not self.projection:
            Ru = Ru + ((G.E(p) - p) / h - 0.5 * (G.E(rn) * mu + rn * G.E(mu)) * self.Dcx) / self.M
            Rv = (Rv + ((G.N(p) - p) / h - 0.5 * (G.N(rn) * mu + rn * G.N(mu)) * self.Dcy) / self.M +
                  self.Fri * self.Ay)
        Ru, Rv = torch.where(self.wu > 0, Ru, u), torch.where(self.wv > 0, Rv, v)
        # constants in p are free: the last mass row (minus the sum of the
        # others) is replaced by p = 0 there
        last = torch.zeros_like(p)
        last[-1, -1] = 1.0
        return torch.stack([Rc, Rm, Ru, Rv, torch.where(last > 0, p, Rp)])

    def newton(self, X):
        """The root near X: Newton's method, each linear system by block
        elimination over the rows (a row couples to its two neighbours)."""
        m2, m1 = X.shape[1:]
        sx = next(d for d in range(3, m1 + 1) if m1 % d == 0 or not self.G.px)
        ii, jj = torch.arange(m1, device=X.device), torch.arange(m2, device=X.device)
        # one product with the Jacobian for each unknown and each cell of a
        # patch sx wide and 3 high: columns so far apart share no row
        colours = [(f, a, b) for f in range(5) for a in range(sx) for b in range(3)]
        seeds = torch.zeros(len(colours), *X.shape, dtype=X.dtype, device=X.device)
        for k, (f, a, b) in enumerate(colours):
            seeds[k, f, b::3, a::sx] = 1.0
        for _ in range(12):
            R = self.residual(X)
            A = torch.zeros(m2, 3, 5, m1, 5, m1, dtype=X.dtype, device=X.device)
            J = torch.func.vmap(lambda e: torch.func.jvp(self.residual, (X,), (e,))[1])(seeds)
            for k, (f, a, b) in enumerate(colours):
                for dj in (-1, 0, 1):
                    js = jj[((jj + dj) % 3 == b) & (jj + dj >= 0) & (jj + dj < m2)]
                    for di in (-1, 0, 1):
                        t = (ii + di) % m1 if self.G.px else ii + di
                        ok = (t % sx == a) & (t >= 0) & (t < m1)
                        A[js[:, None], dj + 1, :, ii[ok][None], f, t[ok][None]] = \
                            J[k][:, js][:, :, ii[ok]].permute(1, 2, 0)
            n = 5 * m1
            A = A.reshape(m2, 3, n, n)
            rhs = -R.permute(1, 0, 2).reshape(m2, n, 1)
            up, y = [], []
            for j in range(m2):
                D, g = A[j, 1], rhs[j]
                if j:
                    D, g = D - A[j, 0] @ up[-1], g - A[j, 0] @ y[-1]
                LU = torch.linalg.lu_factor(D)
                up.append(torch.linalg.lu_solve(*LU, A[j, 2]))
                y.append(torch.linalg.lu_solve(*LU, g))
            for j in range(m2 - 2, -1, -1):
                y[j] = y[j] - up[j] @ y[j + 1]
            dX = torch.stack(y).reshape(m2, 5, m1).permute(1, 0, 2)
            X = X + dX
            size = X.abs().amax((1, 2))
            if bool((dX.abs().amax((1, 2)) <= 1e-11 * size + 1e-300).all()):
                break
        X = X.clone()
        X[4] -= X[4].mean()
        return X


def _exact_steps(case, seed):
    f = scene(case, case["m1"], case["m2"], seed * 1000)
    q = physics(case, case["m1"])
    X = torch.stack([f["c"], f["mu"], f["u"][:, 1:], f["v"][1:], f["p"]])
    for _ in range(case["steps"]):
        S = _Step(q, case["dt"], X, case["path"] == "projection")
        X = S.newton(X)
        u, v = S.velocity(*X)
        X = torch.stack([X[0], X[1], u, v, X[4]])
    c, mu, u, v, p = X
    first = u[:, -1:] if case["periodic"] else torch.zeros_like(u[:, :1])
    out = {"c": c, "mu": mu, "u": torch.cat([first, u], 1),
           "v": torch.cat([torch.zeros_like(v[:1]), v], 0), "p": p}
    return {k: t.cpu().numpy() for k, t in out.items()} if case["host"] else [out]


def _exact_record(case, seed):
    m1, m2 = case["m1"], case["m2"]
    f = scene(case, m1, m2, seed * 1000)
    q = physics(case, m1)
    h, Ly = 1.0 / m1, m2 / m1
    c, u, v = f["c"], f["u"], f["v"]
    S = _Step(q, 1.0, [c, f["mu"], u[:, 1:], v[1:], f["p"]], False)
    r = S.rn
    y = (torch.arange(m2, device=c.device, dtype=c.dtype)[:, None] + 0.5) * h
    eta = _gap(q["rho1"], q["rho2"])
    kin = 0.25 * (u[:, 1:] ** 2 + u[:, :-1] ** 2 + v[1:] ** 2 + v[:-1] ** 2)
    E = r * (kin + 0.5 * q["Cn"] * eta / q["We"] * S.Gn +
             eta / (q["Cn"] * q["We"]) * 0.25 * (c * (c - 1.0)) ** 2 + S.Fri * y)
    div = (u[:, 1:] - u[:, :-1]) / h + (v[1:] - v[:-1]) / h
    lo, hi = c[:-1], c[1:]
    cross = (lo >= 0.5) & (hi < 0.5)
    at = (y[:-1] + h * (lo - 0.5) / torch.where(cross, lo - hi, torch.ones_like(lo)))[cross]
    x = (torch.arange(m1, device=c.device, dtype=c.dtype) + 0.5) * h
    d = {"Vc": (c * 0.5 * (v[1:] + v[:-1])).sum() / c.sum(), "yc": (c * y).sum() / c.sum(),
         "div_max": div.abs().max(), "div_l2": torch.sqrt(h * h * (div * div).sum()),
         "div_expansion": div.max().clamp(min=0.0), "div_compression": (-div).max().clamp(min=0.0),
         "a1": 2.0 / m1 * (h * c.sum(0) * torch.cos(2.0 * math.pi * x)).sum(),
         "y_top": at.max() if len(at) else torch.tensor(0.0),
         "y_bottom": at.min() if len(at) else torch.tensor(Ly)}
    return {"mass": [float(h * h * r.sum()), float(h * h * (r * c).sum())],
            "energy": float(h * h * E.sum()), "diagnostics": {k: float(t) for k, t in d.items()},
            "divergence": div.cpu().numpy()}


def exact(case, seed):
    """What run() returns, from the equations in 64 bits.  None for one outer
    cycle (an iterate, not a solution) and for steps on grids whose Newton
    iteration would take minutes."""
    if case["kind"] == "mass":
        c = scene(case, case["m1"], case["m2"], seed)["c"]
        q = physics(case, case["m1"])
        r = 1.0 / ((q["rho2"] - q["rho1"]) / (q["rho1"] * q["rho2"]) * c + 1.0 / q["rho2"])
        return torch.stack([r.sum(), (r * c).sum()]) / float(case["m1"]) ** 2
    if case["kind"] == "record":
        return _exact_record(case, seed)
    if case["kind"] == "steps" and case["m1"] * case["m2"] * case["m1"] <= 128 * 256 * 128:
        return _exact_steps(case, seed)
    return None
