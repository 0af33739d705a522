"""The oracle's characteristic speeds (Sec. 4.4) against the roots of the
dispersion relation in 60 digits, from rest-frame speeds near that of light to
ones far below it (cold gas, optically thick radiation), where the
discriminant of the quadratic in v cancels down to c^2.  The oracle's inputs
(4-velocity, metric) carry a few rounding errors, of which a boosted
state keeps gamma^2 times as many: 50 * 2^-53 gamma^2 of the speeds' scale.

The oracle is plain FP64 throughout: it is timed as the CPU baseline, and
extended precision is done in software on the hosts that time it."""
import os
from decimal import Decimal, getcontext

import numpy as np
import pytest

from oracle import oracle as O
from paper_1312_6127_gb300 import workloads as W

getcontext().prec = 60


def exact_speeds(gcon, ucon, c2, d):
    D = Decimal
    Au, Bu = D(ucon[d]), D(ucon[0])
    AA, BB, AB = D(gcon[d][d]), D(gcon[0][0]), D(gcon[0][d])
    qa = Bu * Bu - c2 * (BB + Bu * Bu)
    qb = Au * Bu - c2 * (AB + Au * Bu)
    qc = Au * Au - c2 * (AA + Au * Au)
    s = (qb * qb - qa * qc).sqrt()
    return (qb - s) / qa, (qb + s) / qa


@pytest.mark.parametrize("metric", [0, 1])
@pytest.mark.parametrize("cold", [1e-14, 1e-9, 1e-4, 1.0, 1e4])
def test_speeds(metric, cold):
    cfg, x, P = W.random_states(40, seed=11, metric=metric, gamma_max=8.0, magnetised=False, gamma_rad_max=5.0)
    cfg.update(kappa_abs0=0.0, kappa_es0=1.0, n=[8, 8, 8])
    p = O.make_params(cfg)
    P[:, W.UU] = cold * P[:, W.RHO]
    for n in range(len(x)):
        gcov, gcon = O.metric(p, x[n])[:2]
        for d in (1, 2, 3):
            sp = O.flux(p, x[n], d, P[n])[1]
            u = P[n, W.U1:W.U3 + 1]
            alpha = 1.0 / np.sqrt(-gcon[0][0])
            gamma = np.sqrt(1.0 + u @ gcov[1:, 1:] @ u)
            ucon = np.array([gamma / alpha] + [u[i] - gamma * alpha * gcon[0][i + 1] for i in range(3)])
            rho, ug = Decimal(P[n, W.RHO]), Decimal(P[n, W.UU])
            gam = Decimal(cfg["gam"])
            c2 = gam * (gam - 1) * ug / (rho + gam * ug)
            lo, hi = exact_speeds(gcon, ucon, c2, d)
            scale = abs(ucon[d] / ucon[0]) + float(hi - lo) + np.sqrt(gcon[d][d]) * alpha
            tol = 50 * 2.0 ** -53 * gamma ** 2 * scale
            assert abs(float(Decimal(sp[0]) - lo)) <= tol and abs(float(Decimal(sp[1]) - hi)) <= tol, (n, d)


def test_oracle_is_plain_fp64():
    here = os.path.dirname(O.__file__)
    for f in os.listdir(here):
        if f.endswith((".cpp", ".h")):
            assert "long double" not in open(os.path.join(here, f)).read(), f
