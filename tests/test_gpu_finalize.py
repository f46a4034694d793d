"""The finalisation kernels: per-row values against the totals formed without
them (four warps per 32 rows), the rows queued for FP64 recomputation, and a
batch whose member gets other county triangles after the batch was made."""
import numpy as np
import pytest

from paper_2407_11349_gb300 import synth
from paper_2407_11349_gb300.hawkes import HAWKES_F32, HAWKES_F64, HAWKES_LOGLIK_ONLY, Batch, Hawkes

pytestmark = pytest.mark.gpu

P0 = synth.DEFAULT_PARAMS


# less than a warp, one row past a warp and past a block, more rows than one
# step of the grid covers; 5 days put every row near an end of the time range
# (both normal CDFs evaluated), 5,000 days most rows far from both
@pytest.mark.parametrize("n,days", [(1, 100.0), (31, 100.0), (33, 5.0), (129, 5000.0), (4097, 100.0), (60_000, 5000.0)])
def test_rows_add_up_to_the_totals(n, days):
    ds = synth.grid_dataset(n, days, 20, 20, seed=n)
    hk = Hawkes(0).load(ds)
    try:
        for fl in (HAWKES_F64,) if n < 10_000 else (HAWKES_F32,):
            out, rows = hk.loglik_rows(P0, fl)
            ll, g = hk.loglik_grad(P0, fl)
            scale = np.abs(rows[:, :7]).sum(axis=0)
            # FP64 sums of the same n values in another order: n 2^-53 of their
            # absolute sum; the FP32 sweep's atomics add their own order, 1e-9
            tol = (1e-9 if fl == HAWKES_F32 else 4 * n * 2.0 ** -53) * scale + 1e-300
            assert np.all(np.abs(rows[:, :7].sum(axis=0) - out) <= tol)
            assert np.all(np.abs(np.concatenate([[ll], g]) - out) <= tol)
            # ell_i = log lambda_i - Lambda_i
            assert np.allclose(rows[:, 0], rows[:, 7] - rows[:, 8], rtol=1e-14, atol=1e-300)
    finally:
        hk.close()


def test_queued_rows_enter_the_totals_once():
    """Bandwidths so small that rates lie near the FP32 floor: those rows go
    through k_rows64, the others do not, and the totals equal the FP64 path's."""
    ds = synth.grid_dataset(700, 400.0, 20, 20, seed=3)
    p = (0.5, 1.5, 0.7, 0.3, 0.2, 0.5)
    hk = Hawkes(0).load(ds)
    try:
        ref, rows = hk.loglik_rows(p, HAWKES_F64)
        lam_low = rows[:, 7] < -60.0
        assert 0 < lam_low.sum()
        ll, g = hk.loglik_grad(p, HAWKES_F32)
        out, rows32 = hk.loglik_rows(p, HAWKES_F32)
        scale = np.abs(rows[:, 1:7]).sum(axis=0)
        for got in (np.concatenate([[ll], g]), out):
            assert abs(got[0] - ref[0]) <= 1e-6 * abs(ref[0])
            assert np.all(np.abs(got[1:] - ref[1:]) <= 1e-5 * np.maximum(np.abs(ref[1:]), 1e-3 * scale))
        ll1, g1 = hk.loglik_grad(p, HAWKES_F32 | HAWKES_LOGLIK_ONLY)
        assert abs(ll1 - ref[0]) <= 1e-6 * abs(ref[0]) and np.all(np.isnan(g1))
    finally:
        hk.close()


@pytest.mark.parametrize("capture", [False, True])
def test_batch_follows_replaced_counties(capture):
    torch = pytest.importorskip("torch")
    a = synth.grid_dataset(1500, 100.0, 8, 8, seed=1)
    shifted = a.counties.tri_xy.copy()
    shifted[:, 0::2] *= 0.5  # the same counties, half as wide
    hks = [Hawkes(0).load(a) for _ in range(2)]
    dp = torch.tensor(synth.chain_params(2, seed=1), dtype=torch.float64, device="cuda")
    out = torch.zeros((2, 7), dtype=torch.float64, device="cuda")
    b = Batch(hks, [5, 5], [0, 1], HAWKES_F32)
    if capture:
        b.capture(dp.data_ptr(), out.data_ptr())
    torch.cuda.synchronize()
    b.run(dp.data_ptr(), 1, out.data_ptr())
    b.wait()
    hks[1].set_counties(a.counties.tri_county, shifted)
    b.run(dp.data_ptr(), 2, out.data_ptr())
    b.wait()
    got = out.cpu().numpy().copy()
    x, y = hks[1].locations()
    assert x.max() <= 200.0
    for k, h in enumerate(hks):
        h.resample(5, k, 2)
        if k == 1:
            x2, y2 = h.locations()
            assert np.array_equal(x, x2) and np.array_equal(y, y2)
        ref = np.concatenate(h.loglik_grad(dp[k].cpu().numpy(), HAWKES_F32), axis=None)
        assert np.all(np.abs(got[k] - ref) <= 1e-6 * np.abs(ref)), (got[k], ref)
    b.close()
    for h in hks:
        h.close()
