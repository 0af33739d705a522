"""Reconstruction kernels at the sizes where their tiling can go wrong: columns
cut into pieces, rows that cross a warp's 60 cells, the smallest grids, one and
two active directions.  Face fluxes against the oracle at the tolerance of the
other flux tests (1e-10 of |F| plus 1e-3 of its group)."""
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
    dirs = [d for d in (1, 2, 3) if cfg["n"][d - 1] > 1]
    Fo_all = [o.fluxes(e) for e in dirs]
    for d, Fo in zip(dirs, Fo_all):
        err = flux_errors(g.fluxes(d), Fo, group_scales(Fo_all))
        assert err.max() < 1e-10, (d, err.reshape(12, -1).max(axis=1))


@pytest.mark.parametrize("recon,flux", [(W.PPM, W.LAXF), (W.MC, W.HLL)])
@pytest.mark.parametrize("n", [(4, 5, 6), (57, 4, 19), (21, 34, 5), (51, 14, 17), (28, 1, 1), (61, 18, 1)])
def test_box_sizes(n, recon, flux):
    cfg, P = W.minkowski_box(n=n, seed=sum(n), recon=recon, flux=flux)
    check(cfg, P)


@pytest.mark.parametrize("recon", [W.PPM, W.MC])
@pytest.mark.parametrize("n", [(4, 4, 4), (53, 35, 6), (22, 17, 18)])
def test_kerr_schild_sizes(n, recon):
    cfg, P = W.ks_random_state(n=n, seed=sum(n), recon=recon)
    check(cfg, P)
