"""The spatial skip where nothing can be skipped: bandwidths wide enough that
every pair counts, daily ties (whole runs of equal terms), and so many events
that one FP32 sum per row would drift by its rounding bias.

The reference is the FP64 path's totals.  Tolerances as in the parity tests:
log-likelihood 1e-6 relative; each gradient component 1e-5 relative to
max(|g_k|, 1e-3 sum_i |d ell_i / d p_k|)."""
import numpy as np
import pytest

from paper_2407_11349_gb300 import synth
from paper_2407_11349_gb300.hawkes import HAWKES_F32, HAWKES_F64, HAWKES_LOGLIK_ONLY, HAWKES_SKIP_SPATIAL, Hawkes

pytestmark = pytest.mark.gpu


def test_every_pair_kept_at_many_events():
    ds = synth.integer_day_times(synth.grid_dataset(200_000, 1200.0, 60, 60, seed=5))
    p = (0.5, 400.0, 300.0, 0.3, 0.002, 300.0)
    hk = Hawkes(0).load(ds)
    try:
        ref, rows = hk.loglik_rows(p, HAWKES_F64)
        scale = np.abs(rows[:, 1:7]).sum(axis=0)
        ll, g = hk.loglik_grad(p, HAWKES_F32 | HAWKES_SKIP_SPATIAL)
        assert abs(ll - ref[0]) <= 1e-6 * abs(ref[0])
        e = np.abs(g - ref[1:]) / np.maximum(np.abs(ref[1:]), 1e-3 * scale)
        assert np.all(e <= 1e-5), e
        ll1, _ = hk.loglik_grad(p, HAWKES_F32 | HAWKES_SKIP_SPATIAL | HAWKES_LOGLIK_ONLY)
        assert abs(ll1 - ref[0]) <= 1e-6 * abs(ref[0])
    finally:
        hk.close()
