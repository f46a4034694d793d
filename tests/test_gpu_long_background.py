"""A background timescale far longer than the time range: Phi(a) - Phi(b) is a
millionth of either, and the gradient of mu is minus its sum over the events
(background rates are negligible against the excitation's here, but for the first
event's, which has no earlier source).

The reference is the closed form with the error function, 1/2 (erf(a / sqrt 2) -
erf(b / sqrt 2)), added exactly.  Each term is right to a few 2^-53 of itself and
so is a sum of terms of one sign: allowed 1e-13 on the FP64 path; on the FP32 path
the other part (1.3e-6 of it) is right to 1e-6: allowed 1e-11."""
import math

import numpy as np
import pytest

from paper_2407_11349_gb300 import synth
from paper_2407_11349_gb300.hawkes import HAWKES_F32, HAWKES_F64, Hawkes

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("flags,tol", [(HAWKES_F64, 1e-13), (HAWKES_F32, 1e-11)])
def test_gradient_of_mu(flags, tol):
    ds = synth.grid_dataset(2000, 100.0, 20, 20, seed=1)
    mu, tx, tt, th, om, h = p = (1e9, 1e6, 1e8, 1e6, 0.01, 1e4)
    hk = Hawkes(0).load(ds)
    try:
        for g in (hk.loglik_grad(p, flags)[1][0], hk.loglik_rows(p, flags)[1][:, 1].sum()):
            dt = ds.t[:, None] - ds.t[None, :]
            r2 = (ds.x[:, None] - ds.x[None, :]) ** 2 + (ds.y[:, None] - ds.y[None, :]) ** 2
            B = np.where(dt != 0, np.exp(-0.5 * r2 / tx ** 2 - 0.5 * (dt / tt) ** 2), 0.0).sum(axis=1)
            B /= (2 * math.pi) ** 1.5 * tx ** 2 * tt
            E = np.where(dt > 0, np.exp(-om * np.maximum(dt, 0) - 0.5 * r2 / (h * ds.s[None, :]) ** 2), 0.0)
            E = (E / ds.s[None, :] ** 2).sum(axis=1) * om / (2 * math.pi * h * h)
            tail = [0.5 * (math.erf((ds.t[-1] - t) / tt / math.sqrt(2)) + math.erf(t / tt / math.sqrt(2))) for t in ds.t]
            ref = math.fsum(list(B / (mu * B + th * E)) + [-v for v in tail])
            assert abs(g - ref) <= tol * abs(ref), (g, ref)
    finally:
        hk.close()
