"""A batch run inside the caller's own stream capture, right after a member's
county triangles were replaced: the call records itself (no synchronisation) and
the graph evaluates with the new triangles; runs outside the graph do too, before
and after it is launched.  The locations are equal to the bit, the outputs within
1e-6 (the paths differ by the order of FP32 sums)."""
import numpy as np
import pytest

from paper_2407_11349_gb300 import synth
from paper_2407_11349_gb300.hawkes import HAWKES_F32, Batch, Hawkes

pytestmark = pytest.mark.gpu


def test_run_in_the_callers_capture_after_new_counties():
    torch = pytest.importorskip("torch")
    a = synth.grid_dataset(1500, 100.0, 8, 8, seed=1)
    # half as wide, and every triangle many times over: other buffers
    narrow_county, narrow = np.repeat(a.counties.tri_county, 50), np.repeat(a.counties.tri_xy, 50, axis=0)
    narrow[:, 0::2] *= 0.5
    stream = torch.cuda.Stream()
    hks = [Hawkes(0, stream.cuda_stream).load(a) for _ in range(2)]
    dp = torch.tensor(synth.chain_params(2, seed=1), dtype=torch.float64, device="cuda")
    out = torch.zeros((2, 7), dtype=torch.float64, device="cuda")
    b = Batch(hks, [5, 5], [0, 1], HAWKES_F32, stream.cuda_stream)
    torch.cuda.synchronize()

    def check(it):
        torch.cuda.synchronize()
        got = out.cpu().numpy().copy()
        x, y = hks[1].locations()
        for k, h in enumerate(hks):
            h.resample(5, k, it)
            if k == 1:
                assert all(np.array_equal(u, v) for u, v in zip((x, y), h.locations()))
            ref = np.concatenate(h.loglik_grad(dp[k].cpu().numpy(), HAWKES_F32), axis=None)
            assert np.all(np.abs(got[k] - ref) <= 1e-6 * np.abs(ref)), (it, k)

    try:
        b.run(dp.data_ptr(), 1, out.data_ptr())
        check(1)
        hks[1].set_counties(narrow_county, narrow)
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            b.run(dp.data_ptr(), 2, out.data_ptr())
        b.run(dp.data_ptr(), 3, out.data_ptr())  # outside, before the graph has run
        b.wait()
        check(3)
        graph.replay()
        check(2)
        assert hks[1].locations()[0].max() <= 200.0
        hks[1].set_counties(a.counties.tri_county, a.counties.tri_xy)
        b.run(dp.data_ptr(), 4, out.data_ptr())
        b.wait()
        check(4)
        assert hks[1].locations()[0].max() > 200.0
    finally:
        b.close()
        for h in hks:
            h.close()
