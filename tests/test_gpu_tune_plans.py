"""The tuners where variants run one kernel: sizes swept by the column-split kernel
alone keep the first variant whatever the noise of the times, and what they store is
not taken by sizes of the same power of two whose variants differ."""
import json

import pytest

from paper_2407_11349_gb300 import synth
from paper_2407_11349_gb300.hawkes import HAWKES_F32, Batch, Hawkes

pytestmark = pytest.mark.gpu

P0 = synth.DEFAULT_PARAMS


def test_single(tmp_path):
    path = str(tmp_path / "tune.json")
    hk = Hawkes(0)
    try:
        hk.load(synth.grid_dataset(19_000, 1200.0, 40, 40, seed=1))  # n <= 2^15, column split
        if hk.sweep_plan()[0] != 1:
            pytest.skip("another device: 19,000 events are not column split")
        assert hk.tune_cached(P0, path, reps=1) == (0, False)
        assert hk.tune_cached(P0, path, reps=1) == (0, True)
        hk.load(synth.grid_dataset(30_000, 1200.0, 40, 40, seed=1))  # n <= 2^15, row tiles with the band
        assert hk.sweep_plan()[0] == 0
        assert hk.tune_cached(P0, path, reps=1)[1] is False
        assert hk.tune_cached(P0, path, reps=1)[1] is True
        assert len(json.load(open(path))) == 2
    finally:
        hk.close()


def test_batch(tmp_path):
    torch = pytest.importorskip("torch")
    path = str(tmp_path / "tune.json")
    hks = [Hawkes(0).load(synth.grid_dataset(n, 100.0, 20, 20, seed=n)) for n in (700, 900)]
    dp = torch.tensor(synth.chain_params(2, seed=1), dtype=torch.float64, device="cuda")
    out = torch.zeros((2, 7), dtype=torch.float64, device="cuda")
    b = Batch(hks, None, None, HAWKES_F32)
    try:
        torch.cuda.synchronize()
        first = b.tune_cached(dp.data_ptr(), out.data_ptr(), path)
        assert first[0] == 0 and first[3] is False
        assert b.tune_cached(dp.data_ptr(), out.data_ptr(), path)[:4] == (*first[:3], True)
    finally:
        b.close()
        for h in hks:
            h.close()
