"""The work that a user of this library has it do, as cases to measure.

A case is one pass through the public entry points: load the primitives, take
some steps, read the result (``Grid``, ``Batch``), the same from host memory
(``step_host``), a differentiated run (``autograd.steps``), or a point-wise
call.  ``exact`` evaluates the same method in plain torch, 64 bits: the
formulas of the RK3 step (metric, ghost fill, flattened PPM or MC, LAXF or
HLL, flux-CT, geometric source, implicit four-force solve, floors) over whole
arrays, without this library's code.
"""
import math

import numpy as np
import torch

from paper_1312_6127_gb300 import autograd as A
from paper_1312_6127_gb300 import harmrad as H
from paper_1312_6127_gb300 import workloads as W

# flops that one zone needs per sub-step: reconstruction of 12 primitives in 3
# directions (25 each), 3 faces (600), update, source and about 2 residuals of
# the implicit solve (1500)
FLOPS_PER_STAGE = 12 * 3 * 25 + 3 * 600 + 1500


def listed():
    return [
        # the stiff 1D relaxation problem of the tests: nothing but latency
        dict(name="relax_1d_256", kind="relax", n1=256, n2=1, n3=1, steps=20),
        # the tests' torus: a grid that does not fill the GPU
        dict(name="torus_64x32x16", kind="torus", n1=64, n2=32, n3=16, steps=3),
        # an ordinary run written as in the README: g.step(g.cfl_dt())
        dict(name="torus_128x64x32_readme", kind="torus", n1=128, n2=64, n3=32, steps=2, host_dt=True),
        # the paper's fiducial resolution, the headline workload
        dict(name="torus_256x128x64", kind="torus", n1=256, n2=128, n3=64, steps=2),
        # the same with FP32 reconstruction, fluxes and EMFs
        dict(name="torus_256x128x64_split", kind="torus", n1=256, n2=128, n3=64, steps=2, precision=1),
        # the paper's staggered field with the 4-state EMF
        dict(name="torus_128x64x32_uct", kind="torus", n1=128, n2=64, n3=32, steps=2, emf=1),
        # an IMEX integrator
        dict(name="torus_128x64x32_imex2", kind="torus", n1=128, n2=64, n3=32, steps=2, integrator=1),
        # a periodic box of odd sizes, the other reconstruction and flux
        dict(name="box_93x71x45_mc_hll", kind="box", n1=93, n2=71, n3=45, steps=2, recon=1, flux=1),
        # many uneven boxes in one context, optical depths up to 1e6 per cell
        dict(name="batch_12_boxes", kind="batch", count=12, lo=32, hi=64, sizes=4242, steps=1),
        # gradients of a short run with respect to its start and the opacity
        dict(name="adjoint_64x32x16", kind="adjoint", n1=64, n2=32, n3=16, steps=2),
        # point-wise implicit solves from host arrays
        dict(name="zone_implicit_40000", kind="zones", n=40000, metric=1),
        # a step from host memory to host memory
        dict(name="torus_96x64x48_host", kind="host", n1=96, n2=64, n3=48, steps=1),
    ]


def _size(rng, lo, hi, even=False):
    n = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    return n + n % 2 if even else n


def draw(rng):
    kind = rng.choice(["relax", "torus", "torus", "torus", "box", "box", "batch", "adjoint", "zones", "host"])
    if kind == "relax":
        return dict(kind=kind, n1=_size(rng, 32, 4096), n2=1, n3=1, steps=rng.randint(2, 20))
    if kind == "zones":
        return dict(kind=kind, n=_size(rng, 100, 200000), metric=rng.randint(0, 1))
    if kind == "batch":
        return dict(kind=kind, count=rng.randint(2, 24), lo=rng.randint(8, 32), hi=rng.randint(33, 64),
                    sizes=rng.randint(1, 9999), steps=1)
    if kind == "box":
        return dict(kind=kind, n1=_size(rng, 8, 128), n2=_size(rng, 8, 96), n3=_size(rng, 8, 64),
                    steps=rng.randint(1, 3), recon=rng.randint(0, 1), flux=rng.randint(0, 1))
    c = dict(kind=kind, n1=_size(rng, 56, 192), n2=_size(rng, 28, 96), n3=_size(rng, 8, 64, even=True), steps=1)
    if kind == "adjoint":
        c.update(n1=_size(rng, 56, 96), n2=_size(rng, 28, 48), n3=_size(rng, 8, 24, even=True),
                 steps=rng.randint(1, 3))
    elif kind == "torus":
        c.update(steps=rng.randint(1, 3), host_dt=rng.random() < 0.25)
        option = rng.choice(["", "", "precision", "emf", "integrator", "flux"])
        if option:
            c[option] = rng.randint(1, 3) if option == "integrator" else 1
    return c


def _batch_inputs(case, seed):
    """Uneven periodic unit boxes: rho log-normal, speeds up to 0.1, a radiation
    pulse and a per-zone opacity log-uniform in 1e-4 .. 1e6 per cell."""
    gs, g = W.rng(case["sizes"]), W.rng(seed)
    lo, hi = case["lo"], case["hi"]
    gam = 5.0 / 3.0
    T0 = (gam - 1.0) * 1e-2
    cfgs, Ps, Ks = [], [], []
    for _ in range(case["count"]):
        n = [int(round(lo * (hi / lo) ** gs.uniform())) for _ in range(3)]
        shape = n[::-1]
        cfg = W.base_params()
        cfg.update(n=n, dx=[1.0 / m for m in n], gam=gam, a_rad=1e-2 / T0 ** 4, opacity=W.OPAC_FIELD,
                   kappa_es0=0.4)
        P = np.zeros([12] + shape)
        P[W.RHO] = np.exp(g.standard_normal(shape))
        P[W.UU] = 0.01 * P[W.RHO]
        v = g.standard_normal([3] + shape)
        v /= np.linalg.norm(v, axis=0, keepdims=True)
        speed = g.uniform(0.0, 0.1, shape)
        P[W.U1:W.U3 + 1] = v * speed / np.sqrt(1.0 - speed ** 2)
        zc = [(np.arange(m) + 0.5) / m - 0.5 for m in n]
        R2 = zc[2][:, None, None] ** 2 + zc[1][None, :, None] ** 2 + zc[0][None, None, :] ** 2
        P[W.ER] = cfg["a_rad"] * T0 ** 4 * (1.0 + 10.0 * np.exp(-R2 / 0.04))
        cfgs.append(cfg)
        Ps.append(P)
        Ks.append(np.exp(g.uniform(math.log(1e-4), math.log(1e6), shape)) / min(cfg["dx"]))
    return cfgs, Ps, Ks


def _inputs(case, seed):
    """(cfg, P) of a single-grid case."""
    n = (case["n1"], case["n2"], case["n3"])
    if case["kind"] == "relax":
        g = W.rng(seed)
        cfg, P = W.relax_box(n[0], perturb=1e-4 * (1.0 + 0.5 * g.uniform()))
        P[W.ER] *= 1.0 + 0.1 * g.uniform()
    elif case["kind"] == "box":
        cfg, P = W.minkowski_box(n, seed=seed, recon=case["recon"], flux=case["flux"])
    elif case["kind"] == "adjoint":
        cfg, P = W.generic_torus(n, seed=seed)
    else:
        cfg, P = W.torus(n, seed=seed)
        cfg["flux"] = case.get("flux", W.LAXF)
    cfg.update(precision=case.get("precision", 0), emf=case.get("emf", 0), integrator=case.get("integrator", 0))
    return cfg, P


def _zone_inputs(case, seed):
    """Point states in the range of a run's zones and the explicit state one
    update away from them: (cfg, x, U*, guess primitives, h)."""
    n = case["n"]
    cfg, x, P = W.random_states(n, seed=seed, metric=case["metric"], gamma_max=2.0, gamma_rad_max=2.0)
    cfg.update(kappa_abs0=3.0, kappa_es0=1.0)
    g = W.rng(seed + 1)
    P[:, W.RHO] *= 0.1
    P[:, W.B1:W.B3 + 1] *= 0.1
    P[:, W.UU] = P[:, W.RHO] * np.exp(g.uniform(math.log(1e-4), math.log(0.1), n))
    P[:, W.ER] = P[:, W.UU] * np.exp(g.uniform(math.log(1e-2), math.log(10.0), n))
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a))
    geo = _Metric(cfg, t(x[:, 1]), t(x[:, 2]))
    U = _flux(cfg, geo, t(P.T), 0).numpy().T.copy()
    guess = P.copy()
    guess[:, W.UU] *= 1.0 + 0.05 * g.uniform(-1, 1, n)
    guess[:, W.ER] *= 1.0 + 0.05 * g.uniform(-1, 1, n)
    return cfg, x, U, guess, 10.0 ** g.uniform(-4, -2.5, n)


def prepare(case, seed):
    kind = case["kind"]
    s = dict(case=case)
    if kind == "zones":
        s["cfg"], s["x"], s["U"], s["Ps"], s["h"] = _zone_inputs(case, seed)
        return s
    if kind == "batch":
        cfgs, Ps, Ks = _batch_inputs(case, seed)
        s["grid"] = H.Batch(cfgs)
        s["grid"].set_opacity_field(Ks)
        s["P"] = torch.from_numpy(s["grid"].pack(Ps)).cuda()
        return s
    cfg, P = _inputs(case, seed)
    s["grid"] = H.Grid(cfg, precision=cfg["precision"])
    if kind == "host":
        s["P"] = torch.from_numpy(P).pin_memory().numpy()
        s["out"] = torch.empty(P.shape, dtype=torch.float64, pin_memory=True).numpy()
        return s
    s["P"] = torch.from_numpy(P).cuda()
    if kind == "adjoint":
        g = W.rng(seed + 1)
        s["w"] = torch.from_numpy(g.standard_normal(P.shape)).cuda()
        s["kappa"] = cfg["kappa_scale"]
    return s


def run(s):
    case, kind = s["case"], s["case"]["kind"]
    if kind == "zones":
        P, _, _, method = H.zone_implicit(s["cfg"], s["x"], s["U"], s["Ps"], s["h"])
        return dict(P=P, method=method)
    grid = s["grid"]
    if kind == "host":
        grid.step_host(s["P"], s["out"])
        return dict(P=s["out"])
    if kind == "adjoint":
        P0 = s["P"].clone().requires_grad_(True)
        kappa = torch.tensor(s["kappa"], dtype=torch.float64, requires_grad=True)
        P = A.steps(grid, P0, kappa, case["steps"], checkpoint=2)
        (P * s["w"]).sum().backward()
        return dict(P=P.detach(), gP=P0.grad, gkappa=kappa.grad)
    grid.set_prims(s["P"])
    dts = []
    for _ in range(case["steps"]):
        if case.get("host_dt"):
            dts.append(grid.cfl_dt())
            grid.step(dts[-1])
        else:
            grid.step()
    out = dict(P=grid.get_prims(device=True))
    if dts:
        out["dt"] = dts
    return out


def _zones(case):
    if case["kind"] == "zones":
        return case["n"]
    if case["kind"] == "batch":
        g = W.rng(case["sizes"])
        lo, hi = case["lo"], case["hi"]
        return sum(math.prod(int(round(lo * (hi / lo) ** g.uniform())) for _ in range(3))
                   for _ in range(case["count"]))
    return case["n1"] * case["n2"] * case["n3"]


def work(case):
    z = _zones(case)
    if case["kind"] == "zones":  # x, U*, guess, h in; primitives, e_T, steps, method out
        return dict(bytes=z * 8 * (4 + 12 + 12 + 1 + 12 + 1) + 5 * z, flops=z * 1200)
    stages = case["steps"] * (3, 3, 4, 5)[case.get("integrator", 0)]
    nbytes = z * 2 * 12 * 8 + (8 * z if case["kind"] == "batch" else 0)
    if case["kind"] == "adjoint":  # cotangent in, gradient out; a forward step and its transpose
        return dict(bytes=2 * nbytes, flops=3 * z * stages * FLOPS_PER_STAGE)
    return dict(bytes=nbytes, flops=z * stages * FLOPS_PER_STAGE)


# ------------------------------------------------------------------ 64 bits
# Plain torch over whole arrays.  Primitives P[12, ...]; 4-vectors are lists.

def exact(case, seed):
    kind = case["kind"]
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    if kind == "zones":
        cfg, x, U, Ps, h = _zone_inputs(case, seed)
        t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(dev)
        geo = _Metric(cfg, t(x[:, 1]), t(x[:, 2]))
        return dict(P=_implicit(cfg, geo, t(U.T) / geo.gdet, t(Ps.T), t(h)).T.cpu(), method=None)
    if kind == "batch":
        return None  # a zone without a solution takes its neighbours' average: no closed form
    if case.get("emf") or case.get("integrator"):
        return None  # the formulas below are those of the RK3 step with flux-CT
    cfg, P = _inputs(case, seed)
    P, dts = _steps(cfg, torch.from_numpy(P).to(dev), case)
    if kind == "adjoint":  # the gradients of a step with limiters have no closed form
        return dict(P=P, gP=None, gkappa=None)
    return dict(P=P, dt=dts) if case.get("host_dt") else dict(P=P)


class _Metric:
    """Kerr-Schild (or Minkowski) metric in the internal coordinates."""

    def __init__(self, cfg, x1, x2):
        self.mink = cfg["metric"] == 0
        if self.mink:
            one = torch.ones_like(x1 + x2)
            self.g = {(0, 0): -one, (1, 1): one, (2, 2): one, (3, 3): one}
            self.G = dict(self.g)
            self.gdet = self.alpha = one
            return
        a = cfg["a_spin"]
        self.g, self.gdet = _ks_covariant(cfg, x1, x2)
        r = cfg["R0"] + torch.exp(x1)
        th, J2 = _theta(cfg, x2)
        s2 = torch.sin(th) ** 2
        S = r * r + a * a * torch.cos(th) ** 2
        J1, J3 = torch.exp(x1), 2 * math.pi
        tr = 2 * r / S
        self.G = {(0, 0): -(1 + tr), (0, 1): tr / J1, (1, 1): (r * r - 2 * r + a * a) / S / J1 ** 2,
                  (1, 3): a / S / J1 / J3, (2, 2): 1 / S / J2 ** 2, (3, 3): 1 / (S * s2) / J3 ** 2}
        self.alpha = 1 / torch.sqrt(1 + tr)

    @staticmethod
    def _get(m, i, j):
        return m.get((min(i, j), max(i, j)))

    def dn(self, i, j):
        return self._get(self.g, i, j)

    def up(self, i, j):
        return self._get(self.G, i, j)

    def _apply(self, m, v):
        return [sum(self._get(m, i, j) * v[j] for j in range(4) if self._get(m, i, j) is not None) for i in range(4)]

    def lower(self, v):
        return self._apply(self.g, v)

    def raise_(self, v):
        return self._apply(self.G, v)

    def sq3(self, v):
        s = self.dn(1, 1) * v[0] ** 2 + self.dn(2, 2) * v[1] ** 2 + self.dn(3, 3) * v[2] ** 2
        return s if self.mink else s + 2 * self.dn(1, 3) * v[0] * v[2]

    def velocity(self, q):
        """u^mu and u_mu of the ZAMO-relative q^i."""
        gm = torch.sqrt(1 + self.sq3(q))
        u = [gm / self.alpha, q[0], q[1], q[2]]
        if not self.mink:
            u[1] = q[0] - gm * self.alpha * self.up(0, 1)
        return u, self.lower(u)


def _theta(cfg, x2):
    h = cfg["hslope"]
    return (math.pi * x2 + 0.5 * (1 - h) * torch.sin(2 * math.pi * x2),
            math.pi * (1 + (1 - h) * torch.cos(2 * math.pi * x2)))


def _ks_covariant(cfg, x1, x2):
    a = cfg["a_spin"]
    ex = torch.exp(x1)
    r = cfg["R0"] + ex
    th, J2 = _theta(cfg, x2)
    s2 = torch.sin(th) ** 2
    S = r * r + a * a * torch.cos(th) ** 2
    tr = 2 * r / S
    J3 = 2 * math.pi
    g = {(0, 0): tr - 1, (0, 1): tr * ex, (0, 3): -a * tr * s2 * J3, (1, 1): (1 + tr) * ex ** 2,
         (1, 3): -a * s2 * (1 + tr) * ex * J3, (2, 2): S * J2 ** 2,
         (3, 3): s2 * (S + a * a * s2 * (1 + tr)) * J3 ** 2}
    return g, S * torch.abs(torch.sin(th)) * ex * J2 * J3


def _field(geo, u, ul, B):
    bt = B[0] * ul[1] + B[1] * ul[2] + B[2] * ul[3]
    b = [bt] + [(B[i] + bt * u[i + 1]) / u[0] for i in range(3)]
    bl = geo.lower(b)
    return b, bl, sum(x * y for x, y in zip(b, bl))


def _flux(cfg, geo, P, d):
    """sqrt(-g) times the flux along d of the 12 conserved quantities (d = 0:
    the conserved quantities)."""
    u, ul = geo.velocity(P[2:5])
    b, bl, bsq = _field(geo, u, ul, P[5:8])
    ur, url = geo.velocity(P[9:12])
    pg = (cfg["gam"] - 1) * P[1]
    wb, pt = P[0] + P[1] + pg + bsq, pg + 0.5 * bsq
    F = [P[0] * u[d]]
    F += [wb * u[d] * ul[n] - b[d] * bl[n] + (pt if n == d else 0) + (P[0] * u[d] if n == 0 else 0) for n in range(4)]
    F += [P[5 + i] if d == 0 else (P[5 + i] * u[d] - P[4 + d] * u[i + 1]) / u[0] for i in range(3)]
    F += [4 / 3 * P[8] * ur[d] * url[n] + (P[8] / 3 if n == d else 0) for n in range(4)]
    if d:
        F[4 + d] = torch.zeros_like(F[0])
    return geo.gdet * torch.stack(F)


def _opacity(cfg, rho, T):
    if cfg["opacity"] == W.OPAC_KRAMERS:
        ka = cfg["kappa_abs0"] * rho ** 2 * torch.clamp(T, min=cfg["T_kappa_min"]) ** -3.5
    else:
        ka = cfg["kappa_abs0"] * rho
    return cfg["kappa_scale"] * ka, cfg["kappa_scale"] * cfg["kappa_es0"] * rho


def _tau(cfg, geo, P, d):
    ka, ks = _opacity(cfg, P[0], (cfg["gam"] - 1) * P[1] / P[0])
    return (ka + ks) * torch.sqrt(geo.dn(d, d)) * cfg["dx"][d - 1]


def _speeds(geo, u, c2, d):
    AB = 0 if geo.up(0, d) is None else geo.up(0, d)
    a = u[0] ** 2 - c2 * (geo.up(0, 0) + u[0] ** 2)
    b = -2 * (u[d] * u[0] - c2 * (AB + u[d] * u[0]))
    c = u[d] ** 2 - c2 * (geo.up(d, d) + u[d] ** 2)
    s = torch.sqrt(torch.clamp(b * b - 4 * a * c, min=0))
    return (-b - s) / (2 * a), (-b + s) / (2 * a)


def _state_speeds(cfg, geo, P, d):
    u, ul = geo.velocity(P[2:5])
    ur, _ = geo.velocity(P[9:12])
    bsq = _field(geo, u, ul, P[5:8])[2]
    pg = (cfg["gam"] - 1) * P[1]
    w = P[0] + P[1] + pg
    cs2, va2 = cfg["gam"] * pg / w, bsq / (w + bsq)
    g = _speeds(geo, u, torch.clamp(cs2 + va2 - cs2 * va2, 0, 1), d)
    tau = _tau(cfg, geo, P, d)
    r = _speeds(geo, ur, torch.clamp((4 / 3 / tau) ** 2, max=1 / 3), d)
    return g, r


def _along(x, d, o):
    """x at the cells offset by o along direction d (1..3)."""
    return torch.roll(x, -o, dims=-d)


def _ghosts(cfg, P):
    """The 4 ghost zones of every active direction, directions in order."""
    for d in (1, 2, 3):
        n = P.shape[-d]
        if n == 1:
            continue
        parts = [P]
        for side in (0, 1):
            bc = cfg["bc"][2 * (d - 1) + side]
            g = torch.arange(4, device=P.device)
            at = -1 - g if side == 0 else n + g
            src = at % n if bc == W.PERIODIC else at.clamp(0, n - 1)
            if bc == W.POLAR:
                src = g if side == 0 else n - 1 - g
            G = P.index_select(P.dim() - d, src)
            if bc == W.POLAR:
                G = torch.roll(G, -(P.shape[-3] // 2), dims=-3) if P.shape[-3] > 1 else G.clone()
                for q in (1 + d, 4 + d, 8 + d):
                    G[q] = -G[q]
            if bc == W.OUTFLOW:
                for q in (1 + d, 8 + d):
                    G[q] = G[q].clamp(max=0) if side == 0 else G[q].clamp(min=0)
            parts.insert(0, G.flip(-d)) if side == 0 else parts.append(G)
        P = torch.cat(parts, dim=P.dim() - d)
    return P


def _flattener(cfg, P, vg, vr, w, d):
    pg, pr = (cfg["gam"] - 1) * P[1], P[8] / 3

    def f(p, q, v):
        at = lambda o: _along(p, d, o) + w * _along(q, d, o)
        d1, d2, dv = at(1) - at(-1), at(2) - at(-2), _along(v, d, 1) - _along(v, d, -1)
        sp = torch.where(d2 != 0, d1 / d2, torch.zeros_like(d1))
        hit = (d1.abs() > 0.33 * torch.minimum(at(1), at(-1))) & (dv < 0)
        return torch.where(hit, (10 * (sp - 0.75)).clamp(0, 1), torch.zeros_like(d1)), d1 < 0

    (g0, gs), (r0, rs) = f(pg, pr, vg), f(pr, pg, vr)
    fg = torch.maximum(g0, torch.where(gs, _along(g0, d, 1), _along(g0, d, -1)))
    fr = torch.maximum(r0, torch.where(rs, _along(r0, d, 1), _along(r0, d, -1)))
    mx = torch.maximum(fg, fr)
    return torch.stack([(1 - w) * fg + w * mx, (1 - w) * fr + w * mx])


def _slope(s, d):
    dl, dr = s - _along(s, d, -1), _along(s, d, 1) - s
    dc = 0.5 * (_along(s, d, 1) - _along(s, d, -1))
    m = torch.minimum(dc.abs(), 2 * torch.minimum(dl.abs(), dr.abs()))
    return torch.where(dl * dr > 0, torch.sign(dc) * m, torch.zeros_like(m))


def _edges(cfg, s, chi, d):
    D = _slope(s, d)
    if cfg["recon"] == W.MC:
        return s - 0.5 * D, s + 0.5 * D
    lo = 0.5 * (_along(s, d, -1) + s) - (D - _along(D, d, -1)) / 6
    hi = _along(lo, d, 1)
    lo, hi = (1 - chi) * lo + chi * s, (1 - chi) * hi + chi * s
    flat = (hi - s) * (s - lo) <= 0
    dd, m6 = hi - lo, 6 * (s - 0.5 * (lo + hi))
    left, right = dd * m6 > dd * dd, -dd * dd > dd * m6
    L = torch.where(flat, s, torch.where(left, 3 * s - 2 * hi, lo))
    R = torch.where(flat, s, torch.where(right & ~left, 3 * s - 2 * lo, hi))
    return L, R


class _Grid:
    """Metric of the cells and faces of a ghost-inclusive grid, and the steps."""

    def __init__(self, cfg, device):
        self.cfg, self.n = cfg, cfg["n"]
        self.act = [d for d in (1, 2, 3) if self.n[d - 1] > 1]
        self.core = tuple(slice(4, -4) if self.n[d - 1] > 1 else slice(None) for d in (3, 2, 1))

        def x(d, half):
            ng = 4 if self.n[d] > 1 else 0
            i = torch.arange(-ng, self.n[d] + ng, device=device, dtype=torch.float64)
            return cfg["x0"][d] + (i + half) * cfg["dx"][d]

        def at(h1, h2):
            return _Metric(cfg, x(0, h1)[None, None, :], x(1, h2)[None, :, None])

        self.x1, self.x2 = x(0, 0.5)[None, None, :], x(1, 0.5)[None, :, None]
        self.c = at(0.5, 0.5)
        self.f = {1: at(0.0, 0.5), 2: at(0.5, 0.0), 3: self.c}
        if cfg["metric"]:  # d_nu g_{mu kappa} and d_nu sqrt(-g), nu = x1, x2
            y = (self.x1 + 0 * self.x2, self.x2 + 0 * self.x1)
            one, zero = torch.ones_like(y[0]), torch.zeros_like(y[0])
            f = lambda a, b: _ks_covariant(cfg, a, b)
            self.dg = [torch.func.jvp(f, y, t)[1] for t in ((one, zero), (zero, one))]

    def faces(self, P, flat):
        """Face fluxes and largest speeds per direction; flat: flatteners so far."""
        cfg, c = self.cfg, self.c
        u, _ = c.velocity(P[2:5])
        ur, _ = c.velocity(P[9:12])
        F, S = {}, {}
        for d in self.act:
            chi = torch.zeros_like(P[0])
            chi = torch.stack([chi, chi])
            if cfg["recon"] == W.PPM:
                w = torch.clamp(2 * _tau(cfg, c, P, d), max=1)
                chi = _flattener(cfg, P, c.gdet * u[d], c.gdet * ur[d], w, d)
                if d in flat:
                    chi = torch.maximum(chi, flat[d])
                flat[d] = chi
            weight = torch.ones_like(P)
            if cfg["metric"] and d != 2:
                weight[2:8] = c.gdet
                weight[9:12] = c.gdet
            chq = torch.cat([chi[0].expand(8, *P[0].shape), chi[1].expand(4, *P[0].shape)])
            L, R = _edges(cfg, P * weight, chq, d)
            g = self.f[d]
            wf = torch.ones_like(P)
            if cfg["metric"] and d != 2:
                wf[2:8] = g.gdet
                wf[9:12] = g.gdet
            PL, PR = _along(R, d, -1) / wf, L / wf
            (gl, rl), (gr, rr) = _state_speeds(cfg, g, PL, d), _state_speeds(cfg, g, PR, d)
            out = []
            fL, fR, uL, uR = (_flux(cfg, g, X, e) for e in (d, 0) for X in (PL, PR))
            smax = torch.zeros_like(P[0])
            for (l, r), rows in (((gl, gr), slice(0, 8)), ((rl, rr), slice(8, 12))):
                cp = torch.clamp(torch.maximum(l[1], r[1]), min=0)
                cm = torch.clamp(-torch.minimum(l[0], r[0]), min=0)
                if cfg["flux"] == W.LAXF:
                    out.append(0.5 * (fL[rows] + fR[rows] - torch.maximum(cp, cm) * (uR[rows] - uL[rows])))
                else:
                    out.append((cm * fR[rows] + cp * fL[rows] - cm * cp * (uR[rows] - uL[rows])) / (cp + cm))
                smax = torch.maximum(smax, torch.maximum(cp, cm))
            F[d] = torch.cat(out)
            F[d][4 + d] = 0
            if cfg["metric"] and d == 2:
                for side, j in ((2, 4), (3, 4 + self.n[1])):
                    if cfg["bc"][side] == W.POLAR:
                        F[d][:, :, j] = 0
                        smax[:, j] = 0
            S[d] = smax
        for a in self.act:
            for b in self.act:
                if a >= b:
                    continue
                fab, fba = F[a][4 + b].clone(), F[b][4 + a].clone()
                e = 0.25 * (fab + _along(fab, b, -1) - fba - _along(fba, a, -1))
                if cfg["metric"] and 2 in (a, b):
                    for side, j in ((2, 4), (3, 4 + self.n[1])):
                        if cfg["bc"][side] == W.POLAR:
                            e[:, j] = 0
                F[a][4 + b] = 0.5 * (e + _along(e, b, 1))
                F[b][4 + a] = -0.5 * (e + _along(e, a, 1))
        return F, S

    def cfl(self, S):
        v = sum(torch.maximum(S[d], _along(S[d], d, 1)) / self.cfg["dx"][d - 1] for d in self.act)
        return self.cfg["courant"] * float((1 / v[self.core]).min())

    def source(self, P):
        X = torch.zeros_like(P)
        if not self.cfg["metric"]:
            return X
        c = self.c
        u, ul = c.velocity(P[2:5])
        b, bl, bsq = _field(c, u, ul, P[5:8])
        ur, _ = c.velocity(P[9:12])
        pg = (self.cfg["gam"] - 1) * P[1]
        wb, pt = P[0] + P[1] + pg + bsq, pg + 0.5 * bsq
        for k, (dg, dsg) in enumerate(self.dg):
            q = lambda v: sum((1 if i == j else 2) * m * v[i] * v[j] for (i, j), m in dg.items())
            X[2 + k] = 0.5 * c.gdet * (wb * q(u) - q(b)) + pt * dsg
            X[9 + k] = 0.5 * c.gdet * 4 / 3 * P[8] * q(ur) + P[8] / 3 * dsg
        return X

    def step(self, P):
        cfg, flat = self.cfg, {}
        Pa = _ghosts(cfg, P)
        F, S = self.faces(Pa, flat)
        dt = self.cfl(S)
        for s, (A_, B_) in enumerate(((0, 1), (0.75, 0.25), (1 / 3, 2 / 3))):
            if s:
                Pa = _ghosts(cfg, P)
                F, _ = self.faces(Pa, flat)
            U = _flux(cfg, self.c, Pa, 0)
            X = self.source(Pa)
            for d in self.act:
                X = X - (_along(F[d], d, 1) - F[d]) / cfg["dx"][d - 1]
            crop = lambda y: y[(..., *self.core)]
            if s == 0:
                Un = crop(U)
            Us = A_ * Un + B_ * (crop(U) + dt * crop(X))
            geo = _cropped(self.c, self.core, self.n)
            P = _implicit(cfg, geo, Us / geo.gdet, P, torch.full_like(P[0], B_ * dt))
            P = _floors(cfg, geo, P, crop(self.x1.expand(Pa[0].shape)) if cfg["metric"] else None)
        return P, dt


def _cropped(geo, core, n):
    c = _Metric.__new__(_Metric)
    shape = [m + 8 if m > 1 else 1 for m in n[::-1]]
    crop = lambda t: t.expand(shape)[core]
    c.mink = geo.mink
    c.g = {k: crop(v) for k, v in geo.g.items()}
    c.G = {k: crop(v) for k, v in geo.G.items()}
    c.gdet, c.alpha = crop(geo.gdet), crop(geo.alpha)
    return c


def _m1(geo, R, cap):
    """Radiation primitives of R^t_nu (closed form), the energy raised where
    the frame would exceed the Lorentz-factor cap."""
    a = geo.alpha
    up = geo.raise_(R)
    E = a * a * up[0]
    q = [a * (up[i] + (E * geo.up(0, i) if geo.up(0, i) is not None else 0)) for i in (1, 2, 3)]
    q2 = geo.sq3(q)
    s = (4 * cap * cap + 2) / (4 * cap * cap - 1)
    ymax = (4 - s * s) / 3
    y = torch.where(E > 0, q2 / torch.where(E > 0, E * E, torch.ones_like(E)), torch.full_like(E, math.inf))
    over = y > ymax
    E = torch.where(over, 1e-150 + torch.sqrt(torch.where(over, q2, torch.ones_like(q2)) / ymax), E)
    y = torch.where(over, torch.full_like(y, ymax), y)
    s = torch.sqrt(4 - 3 * y)
    f = 1.5 / E / torch.sqrt((s + 2) * (s - 1))
    return [E * (s - 1), f * q[0], f * q[1], f * q[2]]


def _implicit(cfg, geo, U, Ps, h):
    """Solution of T^t_nu - T*^t_nu = h G_nu with rho u^t, B and total
    energy-momentum kept, by Newton's method to round-off."""
    D, T0, B, R0 = U[0], U[1:5], U[5:8], U[8:12]

    def state(x):
        u, ul = geo.velocity(x[1:4])
        rho = D / u[0]
        b, bl, bsq = _field(geo, u, ul, B)
        pg = (cfg["gam"] - 1) * x[0]
        wb, pt = rho + x[0] + pg + bsq, pg + 0.5 * bsq
        T = [wb * u[0] * ul[n] - b[0] * bl[n] + (pt + rho * u[0] if n == 0 else 0) for n in range(4)]
        dT = [T[n] - T0[n] for n in range(4)]
        return u, ul, rho, pg, T, dT, _m1(geo, [R0[n] - dT[n] for n in range(4)], cfg["gamma_rad_max"])

    def error(x, hh):
        u, ul, rho, pg, T, dT, Pr = state(x)
        ur, url = geo.velocity(Pr[1:4])
        Tg = pg / rho
        ka, ks = _opacity(cfg, rho, Tg)
        uru = sum(a * b for a, b in zip(url, u))
        Ru = [4 / 3 * Pr[0] * uru * url[n] + Pr[0] / 3 * ul[n] for n in range(4)]
        uRu = 4 / 3 * Pr[0] * uru ** 2 - Pr[0] / 3
        lam = ka * cfg["a_rad"] * Tg ** 4
        G = [-(ka + ks) * Ru[n] - (ks * uRu + lam) * ul[n] for n in range(4)]
        return torch.stack([dT[n] - hh * G[n] for n in range(4)])

    size = torch.stack([torch.sqrt(geo.up(k, k) - (geo.up(0, k) ** 2 / geo.up(0, 0) if geo.up(0, k) is not None else 0))
                        for k in (1, 2, 3)])
    norm = torch.minimum(T0[0].abs() + (size * T0[1:].abs()).sum(0), R0[0].abs() + (size * R0[1:].abs()).sum(0))

    def far(E):
        e = (E[0].abs() + (size * E[1:].abs()).sum(0)) / norm
        return torch.where(torch.isfinite(e), e, torch.full_like(e, math.inf))

    def newton(x, hh, most):
        best, beste = x, far(error(x, hh))
        for _ in range(most):
            E = error(x, hh)
            J = [torch.func.jvp(lambda y: error(y, hh), (x,), (_unit(x, j),))[1] for j in range(4)]
            M = torch.stack(J, dim=-1).movedim(0, -2)
            scale = M.abs().amax(dim=-2, keepdim=True).clamp(min=1e-300)
            row = (M / scale).abs().amax(dim=-1, keepdim=True).clamp(min=1e-300)
            dx = torch.linalg.solve_ex(M / scale / row, E.movedim(0, -1).unsqueeze(-1) / row)[0]
            dx = (dx / scale.transpose(-1, -2)).squeeze(-1).movedim(-1, 0)
            x = torch.where(torch.isfinite(dx), x - dx, x)
            x = torch.cat([torch.where(x[:1] < 0, -0.5 * x[:1], x[:1]), x[1:]])
            e = far(error(x, hh))
            better = e < beste
            best, beste = torch.where(better, x, best), torch.minimum(e, beste)
            if not bool(better.any()) or float(beste.max()) < 1e-16:
                break
        return best, beste

    x, e = newton(Ps[1:5].clone(), h, 12)
    if float(e.max()) > 1e-9:  # the others: first without the source
        x0, _ = newton(Ps[1:5].clone(), torch.zeros_like(h), 20)
        x1, e1 = newton(x0, h, 20)
        x = torch.where(e1 < e, x1, x)
    u, ul, rho, pg, T, dT, Pr = state(x)
    return torch.stack([rho, x[0], x[1], x[2], x[3], B[0], B[1], B[2], Pr[0], Pr[1], Pr[2], Pr[3]])


def _unit(x, j):
    t = torch.zeros_like(x)
    t[j] = 1
    return t


def _floors(cfg, geo, P, x1):
    P = P.clone()
    for q, cap in ((2, cfg["gamma_gas_max"]), (9, cfg["gamma_rad_max"])):
        g2 = geo.sq3(P[q:q + 3])
        P[q:q + 3] *= torch.where(g2 > cap * cap - 1, torch.sqrt((cap * cap - 1) / g2), torch.ones_like(g2))
    u, ul = geo.velocity(P[2:5])
    bsq = _field(geo, u, ul, P[5:8])[2]
    r = 1.0 if x1 is None else cfg["R0"] + torch.exp(x1)
    P[0] = torch.maximum(P[0], torch.maximum(cfg["floor_rho0"] * r ** cfg["floor_rho_pow"] + 0 * bsq, bsq / cfg["bsq_rho_max"]))
    P[1] = torch.maximum(P[1], torch.maximum(cfg["floor_u0"] * r ** cfg["floor_u_pow"] + 0 * bsq, bsq / cfg["bsq_u_max"]))
    P[0] = torch.maximum(P[0], P[1] / cfg["u_rho_max"])
    return P


def _steps(cfg, P, case):
    grid = _Grid(cfg, P.device)
    dts = []
    for _ in range(case["steps"]):
        P, dt = grid.step(P)
        dts.append(dt)
    return P, dts
