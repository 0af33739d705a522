"""Grids of more than 256 zones per SM at odd sizes: reconstruction and fluxes in
one launch per direction, with the edge values of one direction at a time and full
blocks, which smaller grids (tests/test_gpu_recon.py, test_gpu_faces.py) do not
take.  All faces, and one step, against the oracle at their tolerances (1e-10)."""
import numpy as np
import pytest
import torch

from oracle import oracle as O
from paper_1312_6127_gb300 import harmrad as H
from paper_1312_6127_gb300 import workloads as W
from tests.parity_metrics import flux_errors, group_scales, zone_errors

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("flux", [W.LAXF, W.HLL])
@pytest.mark.parametrize("recon", [W.PPM, W.MC])
@pytest.mark.parametrize("metric,n", [(1, (67, 45, 22)), (0, (93, 45, 17)), (0, (31, 1409, 1))])
def test_fluxes_and_step(metric, n, recon, flux):
    assert np.prod(n) > 256 * torch.cuda.get_device_properties(0).multi_processor_count
    cfg, P = (W.ks_random_state(n=n, seed=41, recon=recon, tau=1.0) if metric
              else W.minkowski_box(n=n, seed=41, recon=recon, vmax=0.1, kappa=(1.0, 1.0)))
    cfg["flux"] = flux
    g = H.Grid(cfg)
    g.set_prims(P)
    o = O.Oracle(cfg)
    o.set_prims(P)
    dirs = [d for d in (1, 2, 3) if n[d - 1] > 1]
    ref = [o.fluxes(d) for d in dirs]
    for d, F in zip(dirs, ref):
        err = flux_errors(g.fluxes(d), F, group_scales(ref))
        assert err.max() < 1e-10, (d, err.reshape(12, -1).max(axis=1))
    dt = o.cfl_dt()
    assert g.cfl_dt() == pytest.approx(dt, rel=1e-12)
    g.step(dt)
    o.step(dt)
    pmhd = (o.status() == 0) & (g.status() == 0)
    e = zone_errors(cfg, g.get_prims(), o.get_prims()).reshape(12, -1)[:, pmhd.ravel()]
    print("%d of %d zones by PMHD, max error %.1e, outcomes differ in %d"
          % (pmhd.sum(), pmhd.size, e.max(), (o.status() != g.status()).sum()))
    assert pmhd.mean() > 0.99 and (o.status() != g.status()).sum() <= 1e-3 * pmhd.size
    assert e.max() < 1e-10, e.max(axis=1)
