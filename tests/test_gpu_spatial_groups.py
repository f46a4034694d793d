"""The spatial skip's row groups of 32: sizes at the edges of a chunk, a tile
and a time window, order built from other locations, parameters and counties
than the evaluation's, far offsets, coincident events, and bandwidths that
keep every pair or none.

The reference is the FP64 path (held to the CPU oracle by the parity tests).
Tolerances as there: log-likelihood 1e-6 relative; each gradient component
1e-5 relative to max(|g_k|, 1e-3 sum_i |d ell_i / d p_k|)."""
import numpy as np
import pytest

from paper_2407_11349_gb300 import synth
from paper_2407_11349_gb300.hawkes import (HAWKES_F32, HAWKES_F64, HAWKES_LOGLIK_ONLY, HAWKES_MODEL1,
                                           HAWKES_SKIP_SPATIAL, Hawkes)

pytestmark = pytest.mark.gpu

P0 = synth.DEFAULT_PARAMS
SP = HAWKES_F32 | HAWKES_SKIP_SPATIAL


def check(hk, p, extra=0, what=""):
    ref, rows = hk.loglik_rows(p, HAWKES_F64 | extra)
    ll, g = hk.loglik_grad(p, SP | extra)
    scale = np.abs(rows[:, 1:7]).sum(axis=0)
    assert abs(ll - ref[0]) <= 1e-6 * abs(ref[0]), (what, ll, ref[0])
    e = np.abs(g - ref[1:]) / np.maximum(np.maximum(np.abs(ref[1:]), 1e-3 * scale), 1e-300)
    assert np.all(e <= 1e-5), (what, e)
    ll1, g1 = hk.loglik_grad(p, SP | extra | HAWKES_LOGLIK_ONLY)
    assert abs(ll1 - ref[0]) <= 1e-6 * abs(ref[0]) and np.all(np.isnan(g1)), what


@pytest.mark.parametrize("n", [1, 31, 32, 33, 255, 257, 2047, 2049, 8193])
def test_sizes_ties_and_windows(n):
    ds = synth.grid_dataset(n, 100.0, 20, 20, seed=300 + n)
    hk = Hawkes(0)
    try:
        for d, extra in ((ds, 0), (synth.integer_day_times(ds), 0), (ds, HAWKES_MODEL1)):
            hk.load(d)
            check(hk, P0, extra, (n, d.name, extra))
        hk.set_spatial_window(256)
        check(hk, P0, 0, (n, "window 256"))
        hk.set_spatial_window(1000)  # not a whole number of tiles
        hk.resample(1, 0, 4)
        check(hk, P0, 0, (n, "window 1000, resampled"))
    finally:
        hk.close()


def test_order_does_not_depend_on_what_built_it():
    """Built without county triangles, at parameters far from those evaluated,
    then moved by a resample."""
    ds = synth.grid_dataset(6000, 100.0, 20, 20, seed=7)
    hk = Hawkes(0)
    try:
        hk.load(ds, counties=False)
        hk.loglik_grad((0.5, 200.0, 0.5, 0.3, 0.2, 2.0), SP)
        hk.set_counties(ds.counties.tri_county, ds.counties.tri_xy)
        for it in range(2):
            hk.resample(3, 0, it)
            for p in (P0, (0.5, 60.0, 3.0, 0.3, 0.05, 6.0), (0.5, 400.0, 90.0, 0.3, 0.01, 300.0)):
                check(hk, p, 0, (it, p))
    finally:
        hk.close()


@pytest.mark.parametrize("shift", [0.0, 2.0e5, -3.0e6])
def test_far_offsets_and_coincident_events(shift):
    """Coordinates and times far from zero against their spread (the boxes are
    widened by the coordinates' FP32 rounding), and many events at one place."""
    ds = synth.grid_dataset(3000, 100.0, 20, 20, seed=8)
    x, y, t = ds.x.copy(), ds.y.copy(), ds.t.copy()
    x[::3], y[::3] = x[0], y[0]
    t[1000:1200] = t[1000]
    hk = Hawkes(0)
    try:
        hk.set_events(t + abs(shift) * 1e-3, ds.county, ds.county_scale, x + shift, y - 0.5 * shift)
        check(hk, P0, 0, shift)
    finally:
        hk.close()
