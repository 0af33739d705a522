"""Adjoint of one step against central differences on the branches that
tests/test_gpu_adjoint.py leaves out: a per-zone opacity field (thin zones and
zones thick enough that the opacity sets the radiation's signal speed), HLL
fluxes and MC slopes on the Kerr-Schild grid.  As there: the Newton tolerance
at round-off, random states far from the limiters' switching points, 1e-6 for
the best of three steps.  kappa_scale, which moves every zone at once: one step
of 1e-5 (below it round-off takes over), 1e-6, or 1e-5 where URAD solves some
zones (accepted at e_T < 1e-9), beside the round-off of the difference:
dL/d kappa_scale is a small remainder of the zones' terms, and a loss that moves
by delta when kappa_scale moves in its last digits (by 1e-14, where the
derivative itself gives 1e-15 or less) leaves delta / h.

The TYPE2 limiter has no case: a limited radiation frame misses R^t_nu by far
more than the 1e-9 at which a solution is accepted, so no solved zone ends
there (random boxes at caps of 1.2, thin to thick: none of 25920 zones)."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1312_6127_gb300 import harmrad as H
from paper_1312_6127_gb300 import workloads as W
from tests.test_gpu_adjoint import TOL, direction

pytestmark = pytest.mark.gpu


def kerr_schild(recon, flux, field):
    cfg, P = W.ks_random_state((24, 14, 8), seed=13, recon=recon, tau=1.0)
    cfg.update(flux=flux, newton_tol=TOL)
    K = None
    if field:
        cfg["opacity"] = W.OPAC_FIELD
        K = 10.0 ** W.rng(14).uniform(-3, 1, P.shape[1:])
    return cfg, P, K


def box(recon, flux):
    cfg, P = W.minkowski_box((8, 9, 7), seed=15, recon=recon, flux=flux)
    cfg.update(opacity=W.OPAC_FIELD, newton_tol=TOL)
    return cfg, P, 10.0 ** W.rng(16).uniform(-2, 3, P.shape[1:])


def thick_zones(cfg, K):
    """Zones whose absorption alone makes tau > 4 / sqrt(3) along x1."""
    p = O.make_params(cfg)
    n = 0
    for k, j, i in np.ndindex(K.shape):
        x = np.array([0.0] + [cfg["x0"][e] + ((i, j, k)[e] + 0.5) * cfg["dx"][e] for e in range(3)])
        n += K[k, j, i] * np.sqrt(O.metric(p, x)[0][1, 1]) * cfg["dx"][0] > 2.31
    return n


CASES = {
    "ks_ppm_hll": lambda: kerr_schild(W.PPM, W.HLL, False),
    "ks_mc_laxf": lambda: kerr_schild(W.MC, W.LAXF, False),
    "ks_mc_hll": lambda: kerr_schild(W.MC, W.HLL, False),
    "ks_ppm_laxf_field": lambda: kerr_schild(W.PPM, W.LAXF, True),
    "ks_ppm_hll_field": lambda: kerr_schild(W.PPM, W.HLL, True),
    "box_ppm_laxf_field": lambda: box(W.PPM, W.LAXF),
    "box_mc_hll_field": lambda: box(W.MC, W.HLL),
}


@pytest.mark.parametrize("name", list(CASES))
def test_adjoint_against_differences(name):
    cfg, P, K = CASES[name]()
    rng = W.rng(17)

    def grid(c, Q):
        g = H.Grid(c)
        if K is not None:
            g.set_opacity_field(K)
        g.set_prims(Q)
        return g

    g = grid(cfg, P)
    dt = g.cfl_dt()
    g.adjoint_enable(True)
    g.step(dt)
    st = g.stats()
    if K is not None:
        assert thick_zones(cfg, K) > 10
    w = rng.standard_normal(P.shape)
    gin, gk = g.step_adjoint(w)

    def loss(c, Q):
        q = grid(c, Q)
        q.step(dt)
        return float((w * q.get_prims()).sum())

    def best(ad, difference, steps, delta=0.0):
        return min((abs(ad - fd) - delta / h) / max(abs(ad), abs(fd)) for h, fd in ((h, difference(h)) for h in steps))

    errs = []
    for _ in range(4):
        v = direction(P, rng)
        errs.append(best(float((gin * v).sum()),
                         lambda h: (loss(cfg, P + h * v) - loss(cfg, P - h * v)) / (2 * h), (1e-5, 1e-6, 1e-7)))
    ks = cfg["kappa_scale"]
    delta = max(abs(loss(dict(cfg, kappa_scale=ks * (1 + e)), P) - loss(cfg, P)) for e in (-2e-14, -1e-14, 1e-14, 2e-14))
    ek = best(gk, lambda h: (loss(dict(cfg, kappa_scale=ks * (1 + h)), P) -
                             loss(dict(cfg, kappa_scale=ks * (1 - h)), P)) / (2 * h * ks), (1e-5,), delta / ks)
    print("%s: urad %d backup %d; directions %s, kappa_scale %.1e beyond a round-off of %.1e in the loss"
          % (name, st["urad_ok"], st["backup"], " ".join("%.1e" % e for e in errs), ek, delta))
    assert max(errs) < 1e-6
    assert ek < (1e-5 if st["urad_ok"] else 1e-6)
