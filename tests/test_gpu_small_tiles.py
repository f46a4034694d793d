"""The column-split sweep (small problems) at the edges of its 128-row and
256-column tiles, of its item lengths and of the rule that hands larger
problems to the row-tile kernel, through every entry point that can take it.

The reference is the row-tile kernel over the same events: one shard that
holds every row (hawkes_shard_moments), finalised by the same kernels.  Both
form each pair term with the same FP32 operations, so they differ by the
order of the sums alone.  Tolerances as in the parity tests: log-likelihood
1e-6 relative; each gradient component 1e-5 relative to max(|g_k|,
1e-3 sum_i |d ell_i / d p_k|)."""
import numpy as np
import pytest

from paper_2407_11349_gb300 import synth
from paper_2407_11349_gb300.hawkes import (HAWKES_BG_TIME, HAWKES_F32, HAWKES_LOGLIK_ONLY,
                                           HAWKES_MODEL1, HAWKES_SKIP_UNDERFLOW, Batch, Hawkes,
                                           hawkes_loglik_grad_noalloc)

pytestmark = pytest.mark.gpu

P0 = synth.DEFAULT_PARAMS


def assert_close(got, ref, rows, what):
    scale = np.abs(rows[:, 1:7]).sum(axis=0)
    assert abs(got[0] - ref[0]) <= 1e-6 * abs(ref[0]), (what, got[0], ref[0])
    e = np.abs(got[1:] - ref[1:]) / np.maximum(np.maximum(np.abs(ref[1:]), 1e-3 * scale), 1e-300)
    assert np.all(e <= 1e-5), (what, e)


def row_tiles(torch, hk, dp, flags):
    m = torch.zeros(6 * hk.n, dtype=torch.float64, device="cuda")
    out = torch.zeros(7, dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    hk.shard_moments(dp.data_ptr(), 0, 1, m.data_ptr(), flags)
    hk.finalize_moments(dp.data_ptr(), m.data_ptr(), out.data_ptr(), flags)
    torch.cuda.synchronize()
    return out.cpu().numpy()


# one row past a row tile, one event short of and past a column tile, the
# first sizes with 2 and 4 column tiles per item, and both sides of the rule's
# line (the last column-split size tried and the first row-tile one)
@pytest.mark.parametrize("n", [129, 511, 513, 9_985, 13_313, 36_865, 65_537])
def test_edges_against_the_row_tile_kernel(n):
    torch = pytest.importorskip("torch")
    ds = synth.grid_dataset(n, 1200.0, 40, 40, seed=n)
    ties = synth.integer_day_times(ds)
    dp = torch.tensor(P0, dtype=torch.float64, device="cuda")
    hk = Hawkes(0)
    try:
        for d, fl in ((ds, 0), (ties, HAWKES_MODEL1), (ties, HAWKES_BG_TIME), (ds, HAWKES_SKIP_UNDERFLOW)):
            hk.load(d)
            ref = row_tiles(torch, hk, dp, fl)
            rows = hk.loglik_rows(P0, HAWKES_F32 | fl)[1]
            got = np.concatenate(hk.loglik_grad(P0, HAWKES_F32 | fl), axis=None)
            assert_close(got, ref, rows, (n, fl))
            ll, g = hk.loglik_grad(P0, HAWKES_F32 | HAWKES_LOGLIK_ONLY | fl)
            assert abs(ll - ref[0]) <= 1e-6 * abs(ref[0]) and np.all(np.isnan(g)), (n, fl)
    finally:
        hk.close()


def test_batch_and_noalloc_take_the_same_tiles():
    torch = pytest.importorskip("torch")
    sizes = [129, 3000, 513, 9_985]
    dss = [synth.grid_dataset(n, 1200.0, 40, 40, seed=n) for n in sizes]
    hks = [Hawkes(0).load(d) for d in dss]
    params = synth.chain_params(len(sizes), seed=1)
    dp = torch.tensor(params, dtype=torch.float64, device="cuda")
    refs = [(row_tiles(torch, h, dp[k], 0), h.loglik_rows(params[k], HAWKES_F32)[1]) for k, h in enumerate(hks)]
    for fl in (0, HAWKES_SKIP_UNDERFLOW):
        out = torch.zeros((len(sizes), 7), dtype=torch.float64, device="cuda")
        b = Batch(hks, None, None, HAWKES_F32 | fl)
        for config in (None, (0, 16, 0), (4, 3, 1)):  # by size, then explicit item lengths
            if config:
                b.set_config(*config)
                assert b.config()[:3] == config
            b.capture(dp.data_ptr(), out.data_ptr())
            torch.cuda.synchronize()
            b.run(dp.data_ptr(), 0, out.data_ptr())
            b.wait()
            for k, o in enumerate(out.cpu().numpy()):
                assert_close(o, *refs[k], (sizes[k], fl, config))
        b.close()
    for k, d in enumerate(dss):
        dev = [torch.tensor(getattr(d, a), dtype=torch.float64, device="cuda") for a in ("t", "x", "y", "s")]
        o = torch.zeros(7, dtype=torch.float64, device="cuda")
        hawkes_loglik_grad_noalloc(*[v.data_ptr() for v in dev], d.n, dp[k].data_ptr(), HAWKES_F32, o.data_ptr(),
                                   torch.cuda.current_stream().cuda_stream)
        torch.cuda.synchronize()
        assert_close(o.cpu().numpy(), *refs[k], (sizes[k], "noalloc"))
    for h in hks:
        h.close()
