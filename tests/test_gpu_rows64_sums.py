"""The FP64 path's sums over many events.  All events at two times under the
time-only background: a row's terms are all equal, which is where a long chain of
additions drifts, and its rate is known in closed form.

Bound on log lambda: no term passes more than about 16 x 16 + n / 256 additions
(16 queues, the rest), an error of 2^-53 each at worst and half of them at most on
the full sum: 440 x 2^-53 = 4.9e-14 at n = 100,000; allowed 5e-14."""
import math

import numpy as np
import pytest

from paper_2407_11349_gb300.hawkes import HAWKES_BG_TIME, HAWKES_F64, HAWKES_MODEL1, Hawkes

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [2_000, 100_000])
def test_equal_terms(n):
    a = n // 3  # events at the first time
    t = np.where(np.arange(n) < a, 10.0, 10.7)
    x = np.linspace(0.0, 1.0, n)
    mu, tx, tt = 0.37, 3.3, 1.1
    hk = Hawkes(0)
    try:
        hk.set_events(t, np.zeros(n, dtype=np.int32), np.ones(1), x, x)
        rows = hk.loglik_rows((mu, tx, tt, 0.0, 0.2, 2.0), HAWKES_F64 | HAWKES_BG_TIME | HAWKES_MODEL1)[1]
        one = math.log(mu) - 0.5 * math.log(2 * math.pi) - 2 * math.log(tx) - math.log(tt) - \
            0.5 * ((10.7 - 10.0) / tt) ** 2
        ref = one + np.log(np.where(np.arange(n) < a, n - a, a).astype(np.float64))
        assert np.all(np.abs(rows[:, 7] - ref) <= 5e-14)
    finally:
        hk.close()
