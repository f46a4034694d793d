"""The rows that the FP32 path recomputes in FP64, where an FP32 bound leaves out
the terms that are exactly zero: sparse events, at scales inside and outside
FP32's range, with and without ties, both models and both backgrounds.

Rows against the CPU oracle: a recomputed row is FP64 throughout, so log lambda
is within 2e-12 of its magnitude where the row is far below the FP32 floor.
Totals against the sum of the rows (the others carry the FP32 error of terms
with exponents near 100, which is not this test's), as in the parity tests
(log-likelihood 1e-6 relative; each gradient component 1e-5 relative to
max(|g_k|, 1e-3 sum_i |d ell_i / d p_k|))."""
import numpy as np
import pytest

import oracle
from paper_2407_11349_gb300.hawkes import HAWKES_BG_TIME, HAWKES_F32, HAWKES_MODEL1, Hawkes

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("unit", [1.0, 1e-15, 1e12])
@pytest.mark.parametrize("flags", [0, HAWKES_MODEL1, HAWKES_BG_TIME])
def test_isolated_events(unit, flags):
    rng = np.random.default_rng(3)
    n = 700
    # pairs of close events, far from all others
    t = np.sort(rng.uniform(1.0, 20000.0, n))
    t[10:14] = t[10]
    x, y = rng.uniform(0, 6000.0, n), rng.uniform(0, 6000.0, n)
    near = np.arange(0, n - 1, 5)
    x[near + 1], y[near + 1] = x[near] + 3.0, y[near] - 2.0
    scale = rng.uniform(0.2, 4.0, 7)
    county = np.arange(n, dtype=np.int32) % 7
    p = (0.5, 20.0 * unit, 7.0, 0.3, 0.2, 2.0 * unit)
    hk = Hawkes(0)
    try:
        hk.set_events(t, county, scale, x * unit, y * unit)
        s = None if flags & HAWKES_MODEL1 else scale[county]
        _, rrows = oracle.loglik_grad(t, x * unit, y * unit, p, s=s, rows=True,
                                        bg_time_only=bool(flags & HAWKES_BG_TIME))
        out, rows = hk.loglik_rows(p, HAWKES_F32 | flags)
        got = np.concatenate(hk.loglik_grad(p, HAWKES_F32 | flags), axis=None)
        far = rrows[:, 7] < np.median(rrows[:, 7]) - 200.0  # below e^-200 of a common rate: recomputed
        assert np.all(np.abs(rows[far, 7] - rrows[far, 7]) <= 2e-12 * np.abs(rrows[far, 7]))
        sc = np.abs(rrows[:, 1:7]).sum(axis=0)
        ref = rows[:, :7].sum(axis=0)
        for o in (out, got):
            assert abs(o[0] - ref[0]) <= 1e-6 * abs(ref[0])
            assert np.all(np.abs(o[1:] - ref[1:]) <= 1e-5 * np.maximum(np.abs(ref[1:]), 1e-3 * sc))
    finally:
        hk.close()
