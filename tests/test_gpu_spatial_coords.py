"""The spatial skip's coordinates carry as many bits as the dense sweep's: two
FP32 words, so a difference is right to 2^-24 of itself and not of the row
group's width.

Clusters of 32 events, far apart in time, at three sites: A and B about one
scaled unit apart at one end of a box almost 8 units wide, a few events at the
other end.  The events of a site share a time (no background among them), so a
row of A has the events of B alone, at one distance.  That distance is the same
in every cluster, so the rows' rates are equal but for its error (their sums of
14 equal terms round alike).  Without excitation the exponent a = r^2 + dt^2
(about 1) is within six roundings of 2^-24 a: an rms of
0.29 sqrt(6) 1.5 2^-24 ln 2 = 4.4e-8 in log lambda; allowed 8e-8.  (One word from
the box's centre, at 2 to 4 units: 2 |d| 2^-23 0.29 sqrt(2) ln 2 = 1.3e-7 more.)"""
import numpy as np
import pytest

from paper_2407_11349_gb300.hawkes import HAWKES_F32, HAWKES_SKIP_SPATIAL, Hawkes

pytestmark = pytest.mark.gpu


def test_differences_inside_a_wide_group():
    rng = np.random.default_rng(11)
    m, tx, tt = 128, 20.0, 7.0
    unit = tx * np.sqrt(2.0 / np.log2(np.e))  # one scaled unit, km
    t, x, y, site = [], [], [], []
    for k in range(m):
        ux, uy = rng.uniform(0.0, 3000.0, 2)
        for s, (d, cnt) in enumerate(((0.0, 14), (0.7, 14), (-7.0, 4))):  # A, B, the other end
            t += [50.0 * tt * (k + 1) + 1e-4 * tt * s] * cnt
            x += [ux + d * unit] * cnt
            y += [uy + d * unit] * cnt
            site += [s] * cnt
    site = np.array(site)
    n = site.size
    p = (0.5, tx, tt, 0.0, 0.2, 2.0)
    hk = Hawkes(0)
    try:
        hk.set_events(np.array(t), np.zeros(n, dtype=np.int32), np.ones(1), np.array(x), np.array(y))
        for flags in (HAWKES_F32 | HAWKES_SKIP_SPATIAL, HAWKES_F32):
            _, rows = hk.loglik_rows(p, flags)
            assert np.std(rows[site < 2, 7]) <= 8e-8, flags
    finally:
        hk.close()
