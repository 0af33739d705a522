"""The Newton continuation queue: a solve that pauses, after `newton_split`
iterations or where it turns to finite differences, and goes on in the queue's
kernel takes the same iterations as one without a pause.  Both kernels evaluate
the same functions; only the compiler's choice of fused operations differs
(1e-15 per evaluation), and a root found to the Newton tolerance 1e-15 moves by
that times the conditioning of the solve, for which 1e-10 is allowed.
"""
import numpy as np
import pytest

from paper_1312_6127_gb300 import harmrad as H
from paper_1312_6127_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def one_step(cfg, P, split):
    g = H.Grid(dict(cfg, newton_tol=1e-15))
    g.set_prims(P)
    g.set_tuning(newton_split=split)
    g.step(g.cfl_dt())
    return g.get_prims(), g.stats()


@pytest.mark.parametrize("split", [1, 3, 5, 50])
@pytest.mark.parametrize("n", [(8, 8, 8), (33, 7, 1)])
def test_paused_solves_end_as_unpaused_ones(n, split):
    cfg, P = W.minkowski_box(n, seed=3, vmax=0.6)
    a, sa = one_step(cfg, P, 0)
    b, sb = one_step(cfg, P, split)
    for k in ("zone_stages", "pmhd_ok", "urad_ok", "backup"):
        assert sa[k] == sb[k], k
    for q in range(12):
        assert np.abs(b[q] - a[q]).max() <= 1e-10 * np.abs(a[q]).max(), q
