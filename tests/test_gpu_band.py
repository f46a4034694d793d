"""The diagonal band of the row-tile sweep: the column-split kernel takes the
columns of each row tile's own rows, and starts while the row tiles run.  Sizes
at a row tile's edge, two kernel variants, batches whose smaller problems have no
column below their rows, captured graphs, calls queued behind one another, and
two contexts at once.

The reference is the same context's row windows, which another kernel sweeps
pair by ordered pair; tolerances as in the parity tests (log-likelihood 1e-6
relative; each gradient component 1e-5 relative to max(|g_k|,
1e-3 sum_i |d ell_i / d p_k|)): the paths differ by the order of the sums
alone."""
import numpy as np
import pytest

from paper_2407_11349_gb300 import synth
from paper_2407_11349_gb300.hawkes import HAWKES_BG_TIME, HAWKES_F32, Batch, Hawkes

pytestmark = pytest.mark.gpu

P0 = synth.DEFAULT_PARAMS


def assert_close(got, ref, rows, what):
    scale = np.abs(rows[:, 1:7]).sum(axis=0)
    assert abs(got[0] - ref[0]) <= 1e-6 * abs(ref[0]), (what, got[0], ref[0])
    e = np.abs(got[1:] - ref[1:]) / np.maximum(np.maximum(np.abs(ref[1:]), 1e-3 * scale), 1e-300)
    assert np.all(e <= 1e-5), (what, e)


def windows(hk, p, flags):
    m = hk.n // 2 + 1
    return sum(np.concatenate(hk.loglik_grad(p, HAWKES_F32 | flags, a, b), axis=None) for a, b in ((0, m), (m, hk.n)))


@pytest.mark.parametrize("n", [32_767, 32_768, 32_769, 49_153])
def test_row_tile_edges_and_variants(n):
    ds = synth.grid_dataset(n, 1200.0, 40, 40, seed=n)
    hk = Hawkes(0)
    try:
        for d, fl in ((ds, 0), (synth.integer_day_times(ds), HAWKES_BG_TIME)):
            hk.load(d)
            for v in (0, 4):  # 2,048 and 1,024 rows per tile
                hk.set_variant(v)
                ref = windows(hk, P0, fl)
                rows = hk.loglik_rows(P0, HAWKES_F32 | fl)[1]
                got = np.concatenate(hk.loglik_grad(P0, HAWKES_F32 | fl), axis=None)
                assert_close(got, ref, rows, (n, fl, v))
    finally:
        hk.close()


def test_batches_and_graphs():
    torch = pytest.importorskip("torch")
    sizes = [700, 2048, 2049, 12_000, 30_000, 36_865]
    hks = [Hawkes(0).load(synth.grid_dataset(n, 1200.0, 40, 40, seed=n)) for n in sizes]
    params = synth.chain_params(len(sizes), seed=1)
    dp = torch.tensor(params, dtype=torch.float64, device="cuda")
    refs = [(windows(h, params[k], 0), h.loglik_rows(params[k], HAWKES_F32)[1]) for k, h in enumerate(hks)]
    b = Batch(hks, None, None, HAWKES_F32)
    try:
        for config in (None, (0, 16, 0), (4, 3, 1)):
            if config:
                b.set_config(*config)
            for captured in (False, True):
                out = torch.zeros((len(sizes), 7), dtype=torch.float64, device="cuda")
                if captured:
                    b.capture(dp.data_ptr(), out.data_ptr())
                torch.cuda.synchronize()
                b.run(dp.data_ptr(), 0, out.data_ptr())
                b.run(dp.data_ptr(), 0, out.data_ptr())
                b.wait()
                for k, o in enumerate(out.cpu().numpy()):
                    assert_close(o, *refs[k], (sizes[k], config, captured))
    finally:
        b.close()
        for h in hks:
            h.close()


def test_queued_calls_and_two_contexts():
    torch = pytest.importorskip("torch")
    n = 36_000
    ds = synth.grid_dataset(n, 1200.0, 40, 40, seed=2)
    params = synth.chain_params(4, seed=3)
    dp = torch.tensor(params, dtype=torch.float64, device="cuda")
    hks = [Hawkes(0).load(ds), Hawkes(0).load(ds)]
    try:
        refs = [(windows(hks[0], params[k], 0), hks[0].loglik_rows(params[k], HAWKES_F32)[1]) for k in range(4)]
        out = torch.zeros((2, 4, 7), dtype=torch.float64, device="cuda")
        torch.cuda.synchronize()
        for k in range(4):
            for c in range(2):  # two streams at once, four calls each without a wait
                hks[c].loglik_grad_async(dp[k].data_ptr(), out[c, k].data_ptr(), HAWKES_F32)
        torch.cuda.synchronize()
        for c in range(2):
            for k in range(4):
                assert_close(out[c, k].cpu().numpy(), *refs[k], (c, k))
    finally:
        for h in hks:
            h.close()
