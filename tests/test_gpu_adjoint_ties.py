"""Adjoint of the limiters at their ties.

Where the state is uniform the limited slopes vanish and the PPM edges lie on
the cell's value.  The derivative taken there is that of the flat cell, for the
MC slopes and the PPM parabola alike, so the two reconstructions have the same
gradient.  Both sum the same terms; only the order of the atomic additions
(about 100 terms an entry) and of the sums over the edges differs, hence
100 * 2^-53 ~ 1e-14 of the largest entry of a variable's gradient, times 100
for cancellation in the steps between.
"""
import numpy as np
import pytest

from paper_1312_6127_gb300 import harmrad as H
from paper_1312_6127_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("flux", [W.LAXF, W.HLL])
@pytest.mark.parametrize("n", [(8, 6, 5), (7, 1, 1), (40, 9, 1)])
def test_uniform_state_has_one_gradient(n, flux):
    out = []
    for recon in (W.MC, W.PPM):
        cfg, P = W.minkowski_box(n, seed=3, recon=recon, flux=flux)
        P[:] = P[:, :1, :1, :1]
        g = H.Grid(dict(cfg, newton_tol=1e-15))
        g.set_prims(P)
        g.adjoint_enable(True)
        g.step(2e-3)
        gP, _ = g.step_adjoint(np.random.default_rng(4).standard_normal(P.shape))
        out.append(np.asarray(gP))
    for q in range(12):
        assert np.abs(out[1][q] - out[0][q]).max() <= 1e-12 * np.abs(out[0][q]).max(), q
