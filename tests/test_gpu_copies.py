"""Primitives and opacity field in and out of a context at ragged sizes: what is
set is what is got, from host and device memory, and any bad value anywhere is
refused."""
import numpy as np
import pytest
import torch

from paper_1312_6127_gb300 import harmrad as H
from paper_1312_6127_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [(4, 1, 1), (5, 4, 7), (33, 17, 1), (64, 9, 31)])
def test_round_trip_and_refusal(n):
    cfg, P = W.minkowski_box(n=n, seed=sum(n))
    g = H.Grid(cfg)
    g.set_prims(P)
    assert np.array_equal(g.get_prims(), P)
    D = torch.from_numpy(P * 1.5).cuda()
    g.set_prims(D)
    assert torch.equal(g.get_prims(device=True), D)
    for q, v in ((W.RHO, 0.0), (W.UU, -1.0), (W.ER, np.nan), (W.UR3, np.inf), (W.B1, -np.inf)):
        bad = P.copy()
        bad[q].flat[-1] = v
        with pytest.raises(H.HarmradError):
            g.set_prims(bad)


@pytest.mark.parametrize("sizes", [[(4, 5, 6), (9, 4, 4)], [(16, 7, 5), (4, 4, 4), (31, 6, 9)]])
def test_batch_round_trip(sizes):
    made = [W.minkowski_box(n=n, seed=3 + i, kappa=(1.0, 1.0)) for i, n in enumerate(sizes)]
    cfgs = [dict(c, opacity=W.OPAC_FIELD) for c, _ in made]
    b = H.Batch(cfgs)
    b.set_prims([P for _, P in made])
    for A, (_, P) in zip(b.get_prims(), made):
        assert np.array_equal(A, P)
    Ks = [np.full(P.shape[1:], 0.5) for _, P in made]
    b.set_opacity_field(Ks)
    Ks[-1].flat[-1] = -1.0
    with pytest.raises(H.HarmradError):
        b.set_opacity_field(Ks)
