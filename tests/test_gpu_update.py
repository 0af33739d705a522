"""One RK3 step of the FP64 update kernel against the oracle over its branches
and ragged sizes: with and without a magnetic field (the gas inversion skips the
field's terms), optically thin (gas inversion as the guess) and thick zones,
every opacity law, one to three active directions, both metrics.  Per-zone
measure below 1e-10, the bound of the other one-step tests, in boxes whose
zones all take the PMHD method."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1312_6127_gb300 import harmrad as H
from paper_1312_6127_gb300 import workloads as W
from tests.parity_metrics import zone_errors

pytestmark = pytest.mark.gpu


def check(cfg, P, K=None):
    g = H.Grid(cfg)
    g.set_prims(P)
    o = O.Oracle(cfg)
    o.set_prims(P)
    if K is not None:
        g.set_opacity_field(K)
        o.set_opacity_field(K)
    dt = o.cfl_dt()
    g.step(dt)
    o.step(dt)
    assert (o.status() == 0).all() and (g.status() == 0).all()
    e = zone_errors(cfg, g.get_prims(), o.get_prims())
    assert e.max() < 1e-10, e.reshape(12, -1).max(axis=1)


@pytest.mark.parametrize("n", [(7, 1, 1), (129, 4, 1), (33, 5, 4)])
@pytest.mark.parametrize("B", [0.0, 0.05])
@pytest.mark.parametrize("kappa,field", [(1e-3, False), (3.0, False), (3.0, True)])
def test_box(n, B, kappa, field):
    cfg, P = W.minkowski_box(n=n, seed=sum(n), B_amp=B, vmax=0.1, kappa=(kappa, kappa))
    K = None
    if field:
        cfg.update(opacity=W.OPAC_FIELD)
        K = kappa * P[W.RHO]
    check(cfg, P, K)


@pytest.mark.parametrize("magnetised", [False, True])
def test_torus(magnetised):
    cfg, P = (W.generic_torus if magnetised else W.torus)((64, 32, 6), seed=3)
    if not magnetised:
        P[W.B1:W.B3 + 1] = 0.0
    check(cfg, P)
