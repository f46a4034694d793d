"""The FP64 pair rows (32 rows per warp, queued columns, table exponential) at
the edges of their groups, segments and row windows, with most pairs exactly
zero and with none, against the CPU oracle.

Both sides are FP64: per-row log lambda, Lambda and partials within 2e-12 of
the sum of their terms' magnitudes (n 2^-53 for the sums, a few 2^-53 times the
exponent, at most 745, for each exponential)."""
import numpy as np
import pytest

import oracle
from paper_2407_11349_gb300 import synth
from paper_2407_11349_gb300.hawkes import HAWKES_BG_TIME, HAWKES_F64, HAWKES_MODEL1, Hawkes

pytestmark = pytest.mark.gpu

P0 = synth.DEFAULT_PARAMS


def check(hk, ds, p, flags):
    s = None if flags & HAWKES_MODEL1 else ds.s
    ref, rrows = oracle.loglik_grad(ds.t, ds.x, ds.y, p, s=s, rows=True, bg_time_only=bool(flags & HAWKES_BG_TIME))
    out, rows = hk.loglik_rows(p, HAWKES_F64 | flags)
    again, rows2 = hk.loglik_rows(p, HAWKES_F64 | flags)
    assert np.array_equal(out, again) and np.array_equal(rows, rows2)  # reproducible to the last bit
    scale = np.maximum(np.abs(rrows), np.abs(rrows).max(axis=0) * 1e-3) + 1e-300
    assert np.all(np.abs(rows[:, 7] - rrows[:, 7]) <= 2e-12 * np.maximum(1.0, np.abs(rrows[:, 7])))
    assert np.all(np.abs(rows[:, :7] - rrows[:, :7]) <= 2e-10 * scale[:, :7])
    assert np.all(np.abs(out - ref) <= 2e-12 * np.maximum(np.abs(ref), np.abs(rrows[:, :7]).sum(axis=0)))
    return ref, rrows


@pytest.mark.parametrize("n", [1, 2, 31, 33, 64, 700, 4100])
@pytest.mark.parametrize("days", [40.0, 4000.0])
def test_groups_segments_and_sparsity(n, days):
    ds = synth.grid_dataset(n, days, 20 if days < 100 else 60, 20 if days < 100 else 60, seed=n)
    hk = Hawkes(0)
    try:
        for d, fl in ((ds, 0), (synth.integer_day_times(ds), HAWKES_MODEL1), (ds, HAWKES_BG_TIME)):
            hk.load(d)
            check(hk, d, P0, fl)
    finally:
        hk.close()


def test_row_windows_and_parameters():
    ds = synth.grid_dataset(1500, 100.0, 20, 20, seed=4)
    hk = Hawkes(0).load(ds)
    try:
        # every pair counts; hardly any excitation does; tiny and huge rates
        for p in (P0, (0.5, 500.0, 90.0, 0.3, 0.01, 300.0), (2.0, 5.0, 2.0, 0.9, 1.5, 0.7)):
            check(hk, ds, p, 0)
            whole = np.concatenate(hk.loglik_grad(p, HAWKES_F64), axis=None)
            edges = [0, 1, 33, 700, 1500]
            parts = [np.concatenate(hk.loglik_grad(p, HAWKES_F64, a, b), axis=None) for a, b in zip(edges, edges[1:])]
            rows = hk.loglik_rows(p, HAWKES_F64)[1]
            assert np.all(np.abs(np.sum(parts, axis=0) - whole) <= 2e-12 * np.abs(rows[:, :7]).sum(axis=0))
    finally:
        hk.close()


@pytest.mark.parametrize("shift", [1.0e5, -4.0e7])
def test_far_from_the_origin(shift):
    """The FP32 bounds take differences from a nearby point: an offset of the
    coordinates does not change which terms are kept."""
    ds = synth.grid_dataset(500, 100.0, 20, 20, seed=5)
    d = synth.Dataset(ds.t, ds.x + shift, ds.y - shift, ds.county, ds.counties, ds.params, "shifted")
    hk = Hawkes(0)
    try:
        hk.set_events(d.t, d.county, d.county_scale, d.x, d.y)
        check(hk, d, P0, 0)
    finally:
        hk.close()


@pytest.mark.parametrize("unit", [1e-21, 1e19])
def test_units(unit):
    """Squares of the coordinates, or the scale factors, outside FP32's range."""
    ds = synth.grid_dataset(300, 100.0, 20, 20, seed=6)
    p = list(P0)
    p[1] *= unit
    p[5] *= unit
    d = synth.Dataset(ds.t, ds.x * unit, ds.y * unit, ds.county, ds.counties, tuple(p), "units")
    hk = Hawkes(0)
    try:
        hk.set_events(d.t, d.county, d.county_scale, d.x, d.y)
        check(hk, d, tuple(p), 0)
    finally:
        hk.close()
