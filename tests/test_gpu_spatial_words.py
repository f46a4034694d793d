"""The spatial skip's coordinates in one and two FP32 words: tight row groups
beside chunks that are too wide for one word, groups too wide themselves, chunk
centres beyond the grid on which their differences are exact, and enough rows
that the tiles are tested in blocks.

The reference is the FP64 path.  A term whose base-2 exponent is a carries the
rounding of three operations on it, 3 a 2^-24 ln 2 with a <= 126: 1.6e-5, and
the sums a few 1e-7 more, so a row's log lambda is within 2e-5; the totals as in
the other tests (log-likelihood 1e-6 relative; each gradient component 1e-5
relative to max(|g_k|, 1e-3 sum_i |d ell_i / d p_k|))."""
import numpy as np
import pytest

from paper_2407_11349_gb300 import synth
from paper_2407_11349_gb300.hawkes import HAWKES_F32, HAWKES_F64, HAWKES_SKIP_SPATIAL, Hawkes

pytestmark = pytest.mark.gpu

P0 = synth.DEFAULT_PARAMS
SP = HAWKES_F32 | HAWKES_SKIP_SPATIAL


def check(hk, p):
    ref, rows = hk.loglik_rows(p, HAWKES_F64)
    out, r32 = hk.loglik_rows(p, SP)
    assert np.all(np.abs(r32[:, 7] - rows[:, 7]) <= 2e-5 * np.maximum(1.0, np.abs(rows[:, 7])))
    scale = np.abs(rows[:, 1:7]).sum(axis=0)
    assert abs(out[0] - ref[0]) <= 1e-6 * abs(ref[0])
    assert np.all(np.abs(out[1:] - ref[1:]) <= 1e-5 * np.maximum(np.abs(ref[1:]), 1e-3 * scale))


@pytest.mark.parametrize("spread", [3.0, 300.0, 3000.0])
def test_clusters_among_scattered_events(spread):
    rng = np.random.default_rng(int(spread))
    n = 4000
    x, y = rng.uniform(0, spread, n), rng.uniform(0, spread, n)
    t = rng.uniform(0.1, 1000.0, n)
    for k in range(4):  # four clusters of 500 events: 10 km, 5 days
        s = slice(500 * k, 500 * k + 500)
        x[s], y[s] = 0.2 * spread * (k + 0.5) + rng.normal(0, 5.0, 500), 0.5 * spread + rng.normal(0, 5.0, 500)
        t[s] = 200.0 * (k + 1) + rng.uniform(0, 5.0, 500)
    o = np.argsort(t)
    hk = Hawkes(0)
    try:
        hk.set_events(t[o], np.arange(n, dtype=np.int32) % 7, rng.uniform(0.2, 4.0, 7), x[o], y[o])
        for p in (P0, (0.5, 5.0, 2.0, 0.3, 1.5, 0.7), (0.5, 80.0, 60.0, 0.3, 0.02, 20.0)):
            check(hk, p)
    finally:
        hk.close()


@pytest.mark.parametrize("shift", [5.0e4, -5.0e6])
def test_centres_beyond_the_exact_grid(shift):
    ds = synth.grid_dataset(3000, 100.0, 20, 20, seed=9)
    hk = Hawkes(0)
    try:
        hk.set_events(ds.t, ds.county, ds.county_scale, 1e-3 * ds.x + shift, 1e-3 * ds.y - shift)
        check(hk, (0.5, 0.02, 7.0, 0.3, 0.2, 0.002))
    finally:
        hk.close()


@pytest.mark.parametrize("days,cells", [(1200.0, 60), (100.0, 20)])
def test_blocks_of_tiles(days, cells):
    ds = synth.grid_dataset(120000, days, cells, cells, seed=10)
    hk = Hawkes(0).load(ds)
    try:
        check(hk, P0)
        hk.resample(2, 0, 1)
        check(hk, P0)
    finally:
        hk.close()
