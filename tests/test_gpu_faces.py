"""FP64 face fluxes over the branches of the face kernel: optically thin to
thick radiation speeds, LAXF and HLL, cold and strongly magnetised gas, fast
flows.  Against the oracle at the tolerance of the other flux tests."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1312_6127_gb300 import harmrad as H
from paper_1312_6127_gb300 import workloads as W
from tests.parity_metrics import flux_errors, group_scales

pytestmark = pytest.mark.gpu


def check(cfg, P):
    g = H.Grid(cfg)
    g.set_prims(P)
    o = O.Oracle(cfg)
    o.set_prims(P)
    Fo_all = [o.fluxes(e) for e in (1, 2, 3)]
    for d in (1, 2, 3):
        err = flux_errors(g.fluxes(d), Fo_all[d - 1], group_scales(Fo_all))
        assert err.max() < 1e-10, (d, err.reshape(12, -1).max(axis=1))
    assert g.cfl_dt() == pytest.approx(o.cfl_dt(), rel=1e-12)


@pytest.mark.parametrize("flux", [W.LAXF, W.HLL])
@pytest.mark.parametrize("tau", [0.0, 1e-3, 2.0, 1e5])
def test_kerr_schild_opacities(tau, flux):
    cfg, P = W.ks_random_state((20, 14, 8), seed=31, tau=tau)
    cfg["flux"] = flux
    check(cfg, P)


@pytest.mark.parametrize("flux", [W.LAXF, W.HLL])
@pytest.mark.parametrize("what", ["cold", "magnetised", "fast", "at_rest"])
def test_box_states(what, flux):
    cfg, P = W.minkowski_box(n=(15, 10, 9), seed=8, flux=flux, vmax=0.98 if what == "fast" else 0.3,
                             B_amp=3.0 if what == "magnetised" else 0.0)
    if what == "cold":
        P[W.UU] = 1e-8 * P[W.RHO]
    if what == "at_rest":
        P[W.U1:W.U3 + 1] = 0.0
        P[W.UR1:W.UR3 + 1] = 0.0
    check(cfg, P)
