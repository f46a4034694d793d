"""Both plans of the symmetric sweep at the edges of their tiles and items and on
both sides of the rule that chooses: the column-split kernel alone, and the row
tiles with the diagonal band.  Each size asserts which plan ran (where the device
has the 152 SMs that the sizes were chosen for).

The reference is two row windows of the same events, which another kernel sweeps
pair by ordered pair (hawkes_shard_moments would run the same row tiles and band);
tolerances as in the parity tests (log-likelihood 1e-6 relative; each gradient
component 1e-5 relative to max(|g_k|, 1e-3 sum_i |d ell_i / d p_k|))."""
import numpy as np
import pytest

from paper_2407_11349_gb300 import synth
from paper_2407_11349_gb300.hawkes import (HAWKES_BG_TIME, HAWKES_F32, HAWKES_LOGLIK_ONLY, HAWKES_MODEL1,
                                           HAWKES_SKIP_UNDERFLOW, Hawkes, HawkesError)

pytestmark = pytest.mark.gpu

P0 = synth.DEFAULT_PARAMS


# column split: one row past an item, one event short of and past a column tile,
# items of 1, 2 and 4 column tiles; with the band: a row tile's edge, a last row tile
# of one row and of nearly all, items of 1, 2, 4 and 8
@pytest.mark.parametrize("n,split,chunk", [(129, 1, 1), (511, 1, 1), (513, 1, 1), (7_937, 1, 2),
                                           (9_985, 1, 2), (13_313, 1, 4), (18_433, 1, 4), (25_001, 1, 4),
                                           (23_999, 0, 4), (28_673, 0, 2), (32_768, 0, 1), (33_793, 0, 8),
                                           (36_865, 0, 1), (65_537, 0, 4)])
def test_edges_of_both_plans(n, split, chunk):
    torch = pytest.importorskip("torch")
    ds = synth.grid_dataset(n, 1200.0, 40, 40, seed=n)
    ties = synth.integer_day_times(ds)
    hk = Hawkes(0)
    try:
        for d, fl in ((ds, 0), (ties, HAWKES_MODEL1), (ties, HAWKES_BG_TIME), (ds, HAWKES_SKIP_UNDERFLOW)):
            hk.load(d)
            if torch.cuda.get_device_properties(0).multi_processor_count == 152:
                assert hk.sweep_plan() == (split, 1 - split, chunk)
            m = n // 2 + 1
            ref = sum(np.concatenate(hk.loglik_grad(P0, HAWKES_F32 | fl, a, b), axis=None) for a, b in ((0, m), (m, n)))
            scale = np.abs(hk.loglik_rows(P0, HAWKES_F32 | fl)[1][:, 1:7]).sum(axis=0)
            ll, g = hk.loglik_grad(P0, HAWKES_F32 | fl)
            assert abs(ll - ref[0]) <= 1e-6 * abs(ref[0]), fl
            assert np.all(np.abs(g - ref[1:]) <= 1e-5 * np.maximum(np.abs(ref[1:]), 1e-3 * scale)), fl
            ll, g = hk.loglik_grad(P0, HAWKES_F32 | HAWKES_LOGLIK_ONLY | fl)
            assert abs(ll - ref[0]) <= 1e-6 * abs(ref[0]) and np.all(np.isnan(g)), fl
    finally:
        hk.close()


def test_no_plan_without_events():
    hk = Hawkes(0)
    try:
        with pytest.raises(HawkesError) as e:
            hk.sweep_plan()
        assert e.value.status == -7
    finally:
        hk.close()
