"""Where a Newton solve pauses changes no byte: the kernel that goes on with it
evaluates the functions of the update kernel that paused it, in FP64 and in
split precision, whose FP32 stages answer a difference in the last bit with up
to 1e-7.  The update kernel with a queue is one kernel for every split, so the
runs below differ in nothing but the kernel an iteration runs in: no tolerance.
(The update kernel without a queue is another one, in which the compiler may
fuse other operations: tests/test_gpu_newton_queue.py.)"""
import numpy as np
import pytest

from paper_1312_6127_gb300 import harmrad as H
from paper_1312_6127_gb300 import workloads as W

pytestmark = pytest.mark.gpu

STATES = {
    "box": lambda: W.minkowski_box((24, 20, 16), seed=3, vmax=0.6),
    "random": lambda: W.ks_random_state((32, 16, 8), seed=9, tau=10.0),
    "torus": lambda: W.torus((64, 32, 16), seed=1),
}


@pytest.mark.parametrize("precision", [H.PREC_FP64, H.PREC_SPLIT])
@pytest.mark.parametrize("state", list(STATES))
def test_split_changes_no_byte(state, precision):
    cfg, P = STATES[state]()
    out = []
    for split in (1, 2, 6, 60):
        g = H.Grid(cfg, precision=precision)
        g.set_prims(P)
        g.set_tuning(newton_split=split)
        g.step()
        out.append((g.get_prims(), g.status(), g.iters(), g.stats()["urad_ok"]))
    assert out[0][2].max() > 6  # solves that a split of 1 or 2 pauses
    for o in out[1:]:
        assert all(np.array_equal(a, b) for a, b in zip(out[0], o))


@pytest.mark.parametrize("precision", [H.PREC_FP64, H.PREC_SPLIT])
def test_split_changes_no_byte_of_a_batch(precision):
    cfgs, Ps, Ks = W.box_batch(3, seed=5, edge=(8, 20))
    out = []
    for split in (1, 3, 6):
        b = H.Batch(cfgs, precision=precision)
        b.set_opacity_field(Ks)
        b.set_prims(Ps)
        b.set_tuning(newton_split=split)
        b.step()
        out.append(b.get_prims())
    for o in out[1:]:
        assert all(np.array_equal(a, b) for a, b in zip(out[0], o))
