"""The FP64 fix-ups of a batch, whose rows are dealt to all blocks whatever
problem they belong to: problems with rows queued for their low rate, with rows
that carry flushed terms, with both and with none, fewer and more problems than
threads in a block, and one problem with invalid parameters among them.

The reference is each problem's own call; tolerances as in the parity tests
(log-likelihood 1e-6 relative; each gradient component 1e-5 relative to
max(|g_k|, 1e-3 sum_i |d ell_i / d p_k|))."""
import numpy as np
import pytest

from paper_2407_11349_gb300 import synth
from paper_2407_11349_gb300.hawkes import HAWKES_F32, Batch, Hawkes, HawkesError

pytestmark = pytest.mark.gpu

LOW = (0.5, 1.5, 0.7, 0.3, 0.2, 0.5)       # rates near the FP32 floor
FLUSHED = (2.0, 5.0, 2.0, 0.9, 1.5, 0.7)   # outputs that rest on flushed terms


def run(sizes, params, invalid=None):
    torch = pytest.importorskip("torch")
    hks = [Hawkes(0).load(synth.grid_dataset(n, 400.0 if k % 2 else 1200.0, 20, 20, seed=k), counties=False)
           for k, n in enumerate(sizes)]
    b = None
    try:
        refs = [(np.concatenate(h.loglik_grad(p, HAWKES_F32), axis=None), h.loglik_rows(p, HAWKES_F32)[1])
                for h, p in zip(hks, params)]
        q = np.array(params, dtype=np.float64)
        if invalid is not None:
            q[invalid, 1] = -1.0
        dp = torch.tensor(q, dtype=torch.float64, device="cuda")
        out = torch.zeros((len(sizes), 7), dtype=torch.float64, device="cuda")
        torch.cuda.synchronize()
        b = Batch(hks, None, None, HAWKES_F32)
        for captured in (False, True):
            if captured:
                b.capture(dp.data_ptr(), out.data_ptr())
            out.zero_()
            torch.cuda.synchronize()
            b.run(dp.data_ptr(), 0, out.data_ptr())
            if invalid is None:
                b.wait()
            else:
                with pytest.raises(HawkesError):
                    b.wait()
            for k, got in enumerate(out.cpu().numpy()):
                if k == invalid:
                    assert np.all(np.isnan(got))
                    continue
                ref, rows = refs[k]
                scale = np.abs(rows[:, 1:7]).sum(axis=0)
                assert abs(got[0] - ref[0]) <= 1e-6 * abs(ref[0]), (k, captured)
                assert np.all(np.abs(got[1:] - ref[1:]) <= 1e-5 * np.maximum(np.abs(ref[1:]), 1e-3 * scale)), (k, captured)
    finally:
        if b is not None:
            b.close()
        for h in hks:
            h.close()


@pytest.mark.parametrize("invalid", [None, 2])
def test_uneven_problems(invalid):
    run([3000, 300, 700, 6000, 1, 500, 257], [LOW, FLUSHED, LOW, FLUSHED, LOW, synth.DEFAULT_PARAMS, LOW], invalid)


def test_more_problems_than_threads_in_a_block():
    sizes = [40 + k % 7 for k in range(300)]
    run(sizes, [(synth.DEFAULT_PARAMS, LOW, FLUSHED)[k % 3] for k in range(300)])
