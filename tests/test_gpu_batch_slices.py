"""Batches of more problems than one launch takes (65,535, the limit of
gridDim.y): the debug build takes 4, so a batch of 11 is staged and finalised in
three launches there.  With resampling, captured and not, one problem with
invalid parameters; against each problem's own call (1e-6 of every output, as the
paths differ by the order of FP32 sums)."""
import os
import subprocess
import sys
import textwrap

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = textwrap.dedent("""
    import numpy as np
    import torch
    from paper_2407_11349_gb300 import synth
    from paper_2407_11349_gb300.hawkes import HAWKES_F32, Batch, Hawkes, HawkesError, hawkes_debug_build
    assert hawkes_debug_build() == 1
    P = 11
    hks = [Hawkes(0).load(synth.grid_dataset(300 + 200 * k, 100.0, 20, 20, seed=k)) for k in range(P)]
    params = synth.chain_params(P, seed=1)
    for bad in (None, 9):
        q = params.copy()
        if bad is not None:
            q[bad, 1] = -1.0
        dp = torch.tensor(q, dtype=torch.float64, device="cuda")
        out = torch.zeros((P, 7), dtype=torch.float64, device="cuda")
        torch.cuda.synchronize()
        b = Batch(hks, [7] * P, list(range(P)), HAWKES_F32)
        for captured in (False, True):
            if captured:
                b.capture(dp.data_ptr(), out.data_ptr())
            b.run(dp.data_ptr(), 3, out.data_ptr())
            try:
                b.wait()
                assert bad is None
            except HawkesError as e:
                assert bad is not None and e.status == -1
            for k, got in enumerate(out.cpu().numpy()):
                if k == bad:
                    assert np.all(np.isnan(got))
                    continue
                hks[k].resample(7, k, 3)
                ref = np.concatenate(hks[k].loglik_grad(params[k], HAWKES_F32), axis=None)
                assert np.all(np.abs(got - ref) <= 1e-6 * np.abs(ref)), (k, captured, got, ref)
        b.close()
    print("SLICES-OK")
""")


def test_more_problems_than_one_launch_takes():
    from paper_2407_11349_gb300 import build as libbuild
    libbuild.build(debug=True)
    r = subprocess.run([sys.executable, "-c", CHILD], cwd=ROOT, env=dict(os.environ, HAWKES_DEBUG="1"),
                       capture_output=True, text=True, timeout=1200)
    assert r.returncode == 0 and "SLICES-OK" in r.stdout, r.stdout[-3000:] + r.stderr[-3000:]
