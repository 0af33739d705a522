"""Grids of one zone: no direction is active, so a step is the implicit solve
(and, on Kerr-Schild, the geometric source) alone.  Every reconstruction and
integrator, one grid and a batch of them, against the oracle at the tolerance
of the other one-step tests (1e-10 in the per-zone measure)."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1312_6127_gb300 import harmrad as H
from paper_1312_6127_gb300 import workloads as W
from tests.parity_metrics import zone_errors

pytestmark = pytest.mark.gpu

DT = 1e-2


def zones(metric, **kw):
    """(cfg, P) of a few single zones of a larger grid."""
    cfg, P = W.minkowski_box((8, 8, 8), seed=3, **kw) if metric == 0 else W.ks_random_state((8, 8, 8), seed=3, **kw)
    out = []
    for z in ((0, 0, 0), (3, 4, 5), (7, 2, 6)):
        x0 = tuple(cfg["x0"][e] + z[2 - e] * cfg["dx"][e] for e in range(3))
        out.append((dict(cfg, n=(1, 1, 1), x0=x0), np.ascontiguousarray(P[(slice(None),) + tuple(slice(i, i + 1) for i in z)])))
    return out


def oracle_step(cfg, P):
    o = O.Oracle(cfg)
    o.set_prims(P)
    o.step(DT)
    return o


@pytest.mark.parametrize("metric", [0, 1])
@pytest.mark.parametrize("recon", [W.PPM, W.MC])
@pytest.mark.parametrize("integrator", [0, 1])
def test_one_zone(metric, recon, integrator):
    for cfg, P in zones(metric, recon=recon):
        cfg = dict(cfg, integrator=integrator)
        g = H.Grid(cfg)
        g.set_prims(P)
        g.step(DT)
        o = oracle_step(cfg, P)
        assert np.array_equal(g.status(), o.status())
        assert zone_errors(cfg, g.get_prims(), o.get_prims()).max() < 1e-10


def test_batch_of_single_zones():
    made = zones(0)
    b = H.Batch([c for c, _ in made])
    b.set_prims([P for _, P in made])
    b.step(DT)
    for (cfg, P), A in zip(made, b.get_prims()):
        assert zone_errors(cfg, A, oracle_step(cfg, P).get_prims()).max() < 1e-10
