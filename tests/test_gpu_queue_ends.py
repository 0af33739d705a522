"""Both ends of the Newton continuation queue are in use, on either metric and
in a batch, and a solve that goes through either ends as without a queue
(tests/test_gpu_newton_queue.py: 1e-10 of a variable's largest value).  With a
split of 60, newton_max's limit, only zones that turn to finite differences
are queued, at one end; with a split of 1 zones pause before they can turn, and
fill the other."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from paper_1312_6127_gb300 import _build
from paper_1312_6127_gb300 import harmrad as H
from paper_1312_6127_gb300 import workloads as W

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def counts(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("queue") / "queue_probe.so")
    subprocess.check_call([_build.nvcc(), "-shared", "-I", _build.CSRC] + _build.ARCH + _build.FLAGS +
                          [os.path.join(HERE, "cuda", "queue_probe.cu"), "-o", so])
    lib = ctypes.CDLL(so)

    def read(g):
        out = (ctypes.c_int * 4)()
        assert lib.queue_counts(g._h, out) == 0
        return list(out)

    return read


def box():
    cfg, P = W.minkowski_box((24, 20, 16), seed=3, vmax=0.6, kappa=(1e4, 1e4))
    g = H.Grid(cfg)
    g.set_prims(P)
    return g


def random_state():
    cfg, P = W.ks_random_state((33, 17, 8), seed=9, tau=10.0)
    g = H.Grid(cfg)
    g.set_prims(P)
    return g


def batch():
    cfgs, Ps, Ks = W.box_batch(3, seed=5, edge=(12, 24))
    b = H.Batch(cfgs)
    b.set_opacity_field(Ks)
    b.set_prims(Ps)
    return b


@pytest.mark.parametrize("make", [box, random_state, batch])
def test_queue_ends(make, counts):
    out = []
    for split in (0, 1, 60):
        g = make()
        g.set_tuning(newton_split=split)
        g.step()
        P = g.get_prims()
        out.append((np.concatenate([p.reshape(12, -1) for p in P], axis=1) if isinstance(P, list)
                    else P.reshape(12, -1), g.stats(), counts(g)))
    (a, sa, qa), (b, sb, qb), (c, sc, qc) = out
    print(qa, qb, qc)
    assert qa[2:] == [0, 0]
    assert qb[2] > 0
    assert qc[2] == 0 and qc[3] > 0
    for other, s in ((b, sb), (c, sc)):
        for k in ("zone_stages", "pmhd_ok", "urad_ok", "backup"):
            assert s[k] == sa[k], k
        for q in range(12):
            assert np.abs(other[q] - a[q]).max() <= 1e-10 * np.abs(a[q]).max(), q
